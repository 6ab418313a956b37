// Elementwise kernels that sit between the Monarch passes of the composite calls: the combination step of the
// complex multiply (further down) and the steps of the feed-forward block's backward pass (Section 4: the block
// is trained by the chain rule through a = M1 x + b1, h = GELU(a), y = M2 h + b2).  The two Monarch backward
// passes are the ordinary monarch_bwd kernels; this file holds what sits between them:
//   mlp_act:   h = GELU(a)                                   (a recomputed by a forward pass of M1)
//   mlp_dact:  da = dh * GELU'(a),  db1 += sum_t da,  db2 += sum_t dy
// Both are pure streaming kernels (16-byte accesses, one pass over their operands).
#include "mma_tiles.cuh"

namespace monarch {
namespace {

constexpr int kThreads = 256;

template <typename T> struct vec16;
template <> struct vec16<float> {
    static constexpr int kElems = 4;
    static __device__ __forceinline__ void load(const float *p, float (&v)[4])
    {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
    static __device__ __forceinline__ void store(float *p, const float (&v)[4])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct vec16<__nv_bfloat16> {
    static constexpr int kElems = 8;
    static __device__ __forceinline__ void load(const __nv_bfloat16 *p, float (&v)[8])
    {
        const uint4 q = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, const float (&v)[8])
    {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<const uint32_t *>(&h2);
        }
        *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// fp32 tensors get the libm-grade forms; bf16 results are rounded to 8 bits of mantissa, so the cheaper forms
// (error <= 5.1e-5) change nothing there and keep both kernels bound by memory rather than by erff / expf
template <typename T> struct act_math;
template <> struct act_math<float> {
    static __device__ __forceinline__ float gelu(float a) { return gelu_erf(a); }
    static __device__ __forceinline__ float grad(float a) { return gelu_erf_grad(a); }
};
template <> struct act_math<__nv_bfloat16> {
    static __device__ __forceinline__ float gelu(float a) { return gelu_fast(a); }
    static __device__ __forceinline__ float grad(float a) { return gelu_fast_grad(a); }
};

// h[t][q] = GELU(a[t][q] (+ b1[q])); n is a multiple of the vector width.  zero1, zero2 (or null): n sums to start from zero
template <typename T>
__global__ void __launch_bounds__(kThreads)
mlp_act_kernel(const T *__restrict__ a, const T *__restrict__ b1, T *__restrict__ h, float *__restrict__ zero1, float *__restrict__ zero2,
               long long vecs, int n)
{
    tc::depend_wait();
    constexpr int V = vec16<T>::kElems, U = 4;          // U independent 16-byte loads in flight per thread
    const long long stride = (long long)gridDim.x * kThreads;
    if (zero1 != nullptr)
        for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < n; i += stride) zero1[i] = zero2[i] = 0.0f;
    for (long long i0 = (long long)blockIdx.x * kThreads + threadIdx.x; i0 < vecs; i0 += U * stride) {
        float v[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * stride < vecs) vec16<T>::load(a + (i0 + u * stride) * V, v[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = i0 + u * stride;
            if (i >= vecs) break;
            if (b1 != nullptr) {
                float b[V];
                vec16<T>::load(b1 + (int)((i * V) % n), b);
#pragma unroll
                for (int e = 0; e < V; ++e) v[u][e] += b[e];
            }
#pragma unroll
            for (int e = 0; e < V; ++e) v[u][e] = act_math<T>::gelu(v[u][e]);
            vec16<T>::store(h + i * V, v[u]);
        }
    }
}

// da = dh * GELU'(a (+ b1)) in place of dh, with the column sums of da (fp32, from the unrounded da) and dy.  Streaming:
// bound by memory as long as the atomic adds stay few, so a CTA takes 32 vectors of columns and a slab of tokens, its 8
// warps every 8th token, and adds their sums in shared memory before the one atomic per column (4096 tokens x 4096 bf16:
// 97 us with one atomic per column for every 8 tokens).
template <typename T>
__global__ void __launch_bounds__(kThreads)
mlp_dact_kernel(T *__restrict__ dh, const T *__restrict__ a, const T *__restrict__ b1, const T *__restrict__ dy,
                float *__restrict__ db1, float *__restrict__ db2, long long tokens, int n, int tokens_per_slab)
{
    constexpr int V = vec16<T>::kElems, kRows = kThreads / 32;
    __shared__ float red[kRows][2][32 * V];
    tc::depend_wait();
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int col = (blockIdx.x * 32 + lane) * V;      // n is a multiple of 256, and of 32 V
    float bias[V], s1[V], s2[V];
#pragma unroll
    for (int e = 0; e < V; ++e) bias[e] = s1[e] = s2[e] = 0.0f;
    if (b1 != nullptr) vec16<T>::load(b1 + col, bias);
    const long long t0 = (long long)blockIdx.y * tokens_per_slab;
    const long long t1 = t0 + tokens_per_slab < tokens ? t0 + tokens_per_slab : tokens;
    // U tokens' loads before the first store: dh is written in place, so the compiler keeps later loads behind a store
    constexpr int U = 4;
    for (long long t = t0 + row; t < t1; t += U * kRows) {
        uint4 g4[U], a4[U], y4[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (t + u * kRows >= t1) break;
            const long long off = (t + u * kRows) * n + col;
            g4[u] = *reinterpret_cast<const uint4 *>(dh + off);
            a4[u] = *reinterpret_cast<const uint4 *>(a + off);
            y4[u] = *reinterpret_cast<const uint4 *>(dy + off);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (t + u * kRows >= t1) break;
            float g[V], av[V], yv[V];
            vec16<T>::load(reinterpret_cast<const T *>(&g4[u]), g);
            vec16<T>::load(reinterpret_cast<const T *>(&a4[u]), av);
            vec16<T>::load(reinterpret_cast<const T *>(&y4[u]), yv);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                g[e] *= act_math<T>::grad(av[e] + bias[e]);
                s1[e] += g[e];
                s2[e] += yv[e];
            }
            vec16<T>::store(dh + (t + u * kRows) * n + col, g);
        }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) {
        red[row][0][lane * V + e] = s1[e];
        red[row][1][lane * V + e] = s2[e];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * 32 * V; i += kThreads) {
        const int which = i / (32 * V), c = i % (32 * V);
        float v[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) v[r] = red[r][which][c];
#pragma unroll
        for (int half = kRows / 2; half > 0; half /= 2)        // pairwise: the fewest roundings
#pragma unroll
            for (int r = 0; r < half; ++r) v[r] += v[r + half];
        atomicAdd((which == 0 ? db1 : db2) + blockIdx.x * 32 * V + c, v[0]);
    }
}

// Combination step of the complex multiply: with A, B, C, D = M(Lr,Rr), M(Li,Ri), M(Lr,Ri), M(Li,Rr) applied to
// the stacked planes [xr; xi] (each [2][plane] elements),
//   y_re = A[0] - B[0] + sgn (C[1] + D[1]),   y_im = A[1] - B[1] - sgn (C[0] + D[0]),
// sgn = -1 for y = M x and +1 for y = M^H x.
template <typename T>
__global__ void __launch_bounds__(kThreads)
cplx_combine_kernel(const T *__restrict__ A, const T *__restrict__ B, const T *__restrict__ C, const T *__restrict__ D,
                    T *__restrict__ y, long long plane_vecs, float sgn)
{
    constexpr int V = vec16<T>::kElems;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < plane_vecs; i += (long long)gridDim.x * kThreads) {
        float a0[V], a1[V], b0[V], b1[V], c0[V], c1[V], d0[V], d1[V], re[V], im[V];
        const long long o0 = i * V, o1 = (plane_vecs + i) * V;
        vec16<T>::load(A + o0, a0); vec16<T>::load(A + o1, a1);
        vec16<T>::load(B + o0, b0); vec16<T>::load(B + o1, b1);
        vec16<T>::load(C + o0, c0); vec16<T>::load(C + o1, c1);
        vec16<T>::load(D + o0, d0); vec16<T>::load(D + o1, d1);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            re[e] = (a0[e] - b0[e]) + sgn * (c1[e] + d1[e]);
            im[e] = (a1[e] - b1[e]) - sgn * (c0[e] + d0[e]);
        }
        vec16<T>::store(y + o0, re);
        vec16<T>::store(y + o1, im);
    }
}

__global__ void merge_status_kernel(unsigned *outer, unsigned *inner)
{
    const unsigned v = *inner;
    if (v != 0) {
        atomicCAS(outer, 0u, v);
        *inner = 0;
    }
}

template <typename T>
int act_t(const void *a, const void *b1, void *h, float *zero1, float *zero2, int64_t tokens, int n, cudaStream_t s)
{
    const long long vecs = (long long)tokens * n / vec16<T>::kElems;
    if (vecs == 0) return MONARCH_OK;
    long long blocks = (vecs + kThreads - 1) / kThreads;
    if (blocks > 148 * 16) blocks = 148 * 16;
    return tc::launch_serialized(mlp_act_kernel<T>, (unsigned)blocks, kThreads, 0, s, (const T *)a, (const T *)b1, (T *)h, zero1, zero2, vecs, n);
}

template <typename T>
int dact_t(void *dh, const void *a, const void *b1, const void *dy, float *db1, float *db2, int64_t tokens, int n,
           cudaStream_t s)
{
    if (tokens == 0) return MONARCH_OK;
    const int bx = n / (32 * vec16<T>::kElems);
    // about 6 CTAs per SM keep enough loads in flight; at least 32 tokens per slab bound the atomics
    long long slabs = (148 * 6 + bx - 1) / bx;
    if (slabs > (tokens + 31) / 32) slabs = (tokens + 31) / 32;
    const int per = (int)((tokens + slabs - 1) / slabs);
    slabs = (tokens + per - 1) / per;
    return tc::launch_serialized(mlp_dact_kernel<T>, dim3((unsigned)bx, (unsigned)slabs), kThreads, 0, s, (T *)dh, (const T *)a, (const T *)b1,
                                 (const T *)dy, db1, db2, (long long)tokens, n, per);
}

}  // namespace

int mlp_act(const void *a, const void *b1, void *h, float *zero1, float *zero2, int64_t tokens, int n, int dtype, cudaStream_t s)
{
    return dtype == MONARCH_F32 ? act_t<float>(a, b1, h, zero1, zero2, tokens, n, s) : act_t<__nv_bfloat16>(a, b1, h, zero1, zero2, tokens, n, s);
}

int mlp_dact(void *dh, const void *a, const void *b1, const void *dy, float *db1, float *db2, int64_t tokens, int n,
             int dtype, cudaStream_t s)
{
    return dtype == MONARCH_F32 ? dact_t<float>(dh, a, b1, dy, db1, db2, tokens, n, s)
                                : dact_t<__nv_bfloat16>(dh, a, b1, dy, db1, db2, tokens, n, s);
}

int cplx_combine(const void *A, const void *B, const void *C, const void *D, void *y, int64_t plane_elems, int adjoint,
                 int dtype, cudaStream_t s)
{
    if (plane_elems == 0) return MONARCH_OK;
    const float sgn = adjoint ? 1.0f : -1.0f;
    const long long vecs = plane_elems / (dtype == MONARCH_F32 ? 4 : 8);
    long long blocks = (vecs + kThreads - 1) / kThreads;
    if (blocks > 148 * 16) blocks = 148 * 16;
    if (dtype == MONARCH_F32)
        cplx_combine_kernel<float><<<(unsigned)blocks, kThreads, 0, s>>>((const float *)A, (const float *)B, (const float *)C,
                                                                        (const float *)D, (float *)y, vecs, sgn);
    else
        cplx_combine_kernel<__nv_bfloat16><<<(unsigned)blocks, kThreads, 0, s>>>(
            (const __nv_bfloat16 *)A, (const __nv_bfloat16 *)B, (const __nv_bfloat16 *)C, (const __nv_bfloat16 *)D,
            (__nv_bfloat16 *)y, vecs, sgn);
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

int merge_status(unsigned *outer, unsigned *inner, cudaStream_t s)
{
    merge_status_kernel<<<1, 1, 0, s>>>(outer, inner);
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

}  // namespace monarch
