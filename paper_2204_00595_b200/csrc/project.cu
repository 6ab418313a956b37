// Conversions between a dense n x n matrix and the Monarch factors (n = m*m):
//   monarch_dense    Eq. (2):       M[l*m+j][k*m+i] = L[j][l][k] R[k][j][i]
//   monarch_project  Algorithm 1:   view A as A~[l][j][k][i] = A[l*m+j][k*m+i]; for every (j, k) replace the m x m
//                                   slice A~[:, j, k, :] by its best rank-1 approximation sigma u v^T and store
//                                   L[j][:, k] = sqrt(sigma) u,  R[k][j][:] = sqrt(sigma) v.
// The m*m slices are independent: one CTA per slice.  Only the leading singular triplet is needed, so
// leading_pair_kernel iterates for that one vector and never forms the rest of the decomposition; a caller that asks
// for the number of plane rotations gets jacobi_kernel, the full one-sided Jacobi iteration that performs them.
// Arithmetic is fp32 whatever the storage dtype.
#include <type_traits>

#include "common.cuh"

namespace monarch {
namespace {

// Bound by the n*n elements written.  A CTA keeps a column range of R~_j (j fixed) in registers, 16 bytes per access,
// and writes it scaled by L[j][l][k] for kDenseRows rows l, so that R is read m / kDenseRows times instead of m times
// and every store is 16 bytes (n = 4096 fp32: 30.6 us with one scalar store per element and thread).
constexpr int kDenseRows = 16, kDenseVecs = 4;

template <typename T>
__global__ void __launch_bounds__(256)
dense_kernel(const T *__restrict__ L, const T *__restrict__ R, T *__restrict__ M, int m)
{
    constexpr int V = 16 / sizeof(T);
    const int j = blockIdx.x, l0 = blockIdx.y * kDenseRows, n = m * m;
    const int c0 = (blockIdx.z * kDenseVecs * 256 + threadIdx.x) * V;
    float r[kDenseVecs][V];
#pragma unroll
    for (int q = 0; q < kDenseVecs; ++q) {
        const int col = c0 + q * 256 * V;
        if (col < n) {
            const uint4 raw = *reinterpret_cast<const uint4 *>(R + ((size_t)(col / m) * m + j) * m + col % m);
#pragma unroll
            for (int e = 0; e < V; ++e) r[q][e] = elem<T>::load(reinterpret_cast<const T *>(&raw) + e);
        }
    }
#pragma unroll 4
    for (int l = l0; l < l0 + kDenseRows; ++l) {
#pragma unroll
        for (int q = 0; q < kDenseVecs; ++q) {
            const int col = c0 + q * 256 * V;
            if (col >= n) continue;
            const float w = elem<T>::load(L + ((size_t)j * m + l) * m + col / m);
            uint4 raw;
#pragma unroll
            for (int e = 0; e < V; ++e) elem<T>::store(reinterpret_cast<T *>(&raw) + e, w * r[q][e]);
            *reinterpret_cast<uint4 *>(M + ((size_t)l * m + j) * n + col) = raw;
        }
    }
}

constexpr int kMaxSweeps = 30;
// columns count as orthogonal below this cosine: a few times the rounding noise of an fp32 dot product of m terms
constexpr float kOrthoTol = 2e-6f;

// One-sided Jacobi in shared memory: columns are rotated in pairs until they are mutually orthogonal; their norms are
// then the singular values and the normalised columns the left singular vectors; v = S^T u / sigma is one more pass
// over the slice.  `rotations` counts the plane rotations.  A column pair is handled by G lanes (m/G rows each): G = 8 for m <= 64, so that a warp rotates four pairs at once
// - with 64-element columns a whole warp per pair would spend most of its instructions on shuffle and scalar work
// replicated over 32 lanes - and G = 32 for m = 128, where the strided rows of four different columns would
// collide in the shared-memory banks.  Several CTAs share an SM.
template <int M> struct ProjectCfg {
    static constexpr int kG = M >= 128 ? 32 : 8;
    static constexpr int kPairsPerPass = 32 / kG;                       // pairs a warp rotates at once
    static constexpr int kWarps = M >= 128 ? 32 : (M / 8 < 2 ? 2 : M / 8);
    static constexpr int kPasses = (M / 2) / (kWarps * kPairsPerPass);  // passes per round
};

template <typename T, int M>
__global__ void __launch_bounds__(ProjectCfg<M>::kWarps * 32)
jacobi_kernel(const T *__restrict__ A, T *__restrict__ L, T *__restrict__ R, unsigned long long *rotations)
{
    using C = ProjectCfg<M>;
    constexpr int N = M * M;
    constexpr int kWarps = C::kWarps, G = C::kG;
    static_assert(kWarps * C::kPairsPerPass * C::kPasses == M / 2, "a round covers every column once");
    constexpr int kPitch = M + 1;                         // column pitch in floats (odd: no bank conflicts)
    constexpr int kRows = M / G;                          // rows per lane
    extern __shared__ float cols[];                       // cols[i * kPitch + l] = S[l][i]
    __shared__ float red_val[32];
    __shared__ int red_idx[32];
    __shared__ float u_s[M];
    __shared__ float sigma_s;
    __shared__ int best_s;

    const int j = blockIdx.x / M, k = blockIdx.x % M;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane / G, sub = lane % G;
    const T *slice = A + (size_t)j * N + (size_t)k * M;   // element (l, i) at slice[l * M * N + i]

    for (int e = threadIdx.x; e < M * M; e += kWarps * 32) {
        const int l = e / M, i = e % M;
        cols[i * kPitch + l] = elem<T>::load(slice + (size_t)l * M * N + i);
    }
    __syncthreads();

    unsigned my_rot = 0;
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        int rotated = 0;
        for (int rr = 0; rr < M - 1; ++rr) {
#pragma unroll
            for (int pass = 0; pass < C::kPasses; ++pass) {
                // round-robin tournament: column M-1 stays, the others move round a circle of M-1 seats
                const int p = (warp * C::kPasses + pass) * C::kPairsPerPass + grp;
                int ca = rr + p, cb = rr - p + (M - 1);
                if (ca >= M - 1) ca -= M - 1;
                if (cb >= M - 1) cb -= M - 1;
                if (p == 0) ca = M - 1;
                float *a = cols + ca * kPitch + sub, *b = cols + cb * kPitch + sub;
                float av[kRows], bv[kRows];
                float aa = 0.0f, bb = 0.0f, ab = 0.0f;
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    av[q] = a[G * q];
                    bv[q] = b[G * q];
                    aa = fmaf(av[q], av[q], aa);
                    bb = fmaf(bv[q], bv[q], bb);
                    ab = fmaf(av[q], bv[q], ab);
                }
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) {
                    aa += __shfl_xor_sync(0xffffffffu, aa, o);
                    bb += __shfl_xor_sync(0xffffffffu, bb, o);
                    ab += __shfl_xor_sync(0xffffffffu, ab, o);
                }
                // rotate unless the two columns are already orthogonal to working precision.  The angle only has to
                // be roughly right (orthogonality is re-tested every sweep, and the factors are formed from a
                // re-normalised column), so the fast reciprocal / square-root forms are enough.
                if (ab * ab > (kOrthoTol * kOrthoTol) * (aa * bb)) {
                    // clamped: columns that are pure rounding noise (rank-deficient slices) give huge ratios
                    const float zeta = fmaxf(fminf(__fdividef(bb - aa, 2.0f * ab), 1e15f), -1e15f);
                    const float w = fmaf(zeta, zeta, 1.0f);
                    const float t = copysignf(__fdividef(1.0f, fabsf(zeta) + w * rsqrtf(w)), zeta);
                    const float c = rsqrtf(fmaf(t, t, 1.0f)), s = c * t;
#pragma unroll
                    for (int q = 0; q < kRows; ++q) {
                        a[G * q] = c * av[q] - s * bv[q];
                        b[G * q] = s * av[q] + c * bv[q];
                    }
                    rotated = 1;
                    if (sub == 0) ++my_rot;
                }
            }
            __syncthreads();
        }
        if (!__syncthreads_or(rotated)) break;
    }
    if (my_rot) atomicAdd(rotations, (unsigned long long)my_rot);

    // the column of largest norm carries sigma_1 u_1
    float best = -1.0f;
    int best_i = 0;
    for (int i = threadIdx.x; i < M; i += kWarps * 32) {
        float s2 = 0.0f;
        for (int l = 0; l < M; ++l) s2 = fmaf(cols[i * kPitch + l], cols[i * kPitch + l], s2);
        if (s2 > best) { best = s2; best_i = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        if (ov > best || (ov == best && oi < best_i)) { best = ov; best_i = oi; }
    }
    if (lane == 0) { red_val[warp] = best; red_idx[warp] = best_i; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float bv = red_val[0];
        int bi = red_idx[0];
        for (int w = 1; w < kWarps; ++w)
            if (red_val[w] > bv || (red_val[w] == bv && red_idx[w] < bi)) { bv = red_val[w]; bi = red_idx[w]; }
        sigma_s = sqrtf(fmaxf(bv, 0.0f));
        best_s = bi;
    }
    __syncthreads();
    const float sigma = sigma_s, root = sqrtf(sigma);
    const float inv = sigma > 0.0f ? 1.0f / sigma : 0.0f;
    for (int l = threadIdx.x; l < M; l += kWarps * 32) {
        const float ul = cols[best_s * kPitch + l] * inv;
        u_s[l] = ul;
        elem<T>::store(L + ((size_t)j * M + l) * M + k, root * ul);
    }
    __syncthreads();
    // v = S^T u / sigma from the original slice (the shared copy has been rotated), scaled by sqrt(sigma)
    for (int i = threadIdx.x; i < M; i += kWarps * 32) {
        float acc = 0.0f;
        for (int l = 0; l < M; ++l) acc = fmaf(elem<T>::load(slice + (size_t)l * M * N + i), u_s[l], acc);
        elem<T>::store(R + ((size_t)k * M + j) * M + i, root * acc * inv);
    }
}

template <typename T, int M>
int launch_jacobi(const void *A, void *L, void *R, unsigned long long *rotations, cudaStream_t s)
{
    constexpr int kWarps = ProjectCfg<M>::kWarps;
    constexpr int smem = M * (M + 1) * (int)sizeof(float);
    static bool attr = false;
    if (!attr && smem > 48 * 1024) {
        MONARCH_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel<T, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr = true;
    }
    jacobi_kernel<T, M><<<M * M, kWarps * 32, smem, s>>>((const T *)A, (T *)L, (T *)R, rotations);
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

// ---- leading singular pair of a slice ------------------------------------------------------------------------------
//  1. Power iteration on S^T S from TWO fixed unrelated start vectors.  It has converged when the two agree and have
//     stopped moving, to kPowerTol: neither alone would show a start vector that happens to be orthogonal to v_1.  Two that
//     stand still and differ are eigenvectors both: singular values that are equal to rounding, or one vector that is
//     orthogonal to v_1; the one with the larger singular value is taken.
//     At most kPowerSteps steps are spent on it, enough for (sigma_2 / sigma_1)^2 up to about 0.7.
//     a. Where the two are within kNear of one another after four steps and every step leaves less than kFast of it, both go on
//        with S^T S - shift I and are tested every other step.  The shift is half of what the rate says of sigma_2^2, which brings
//        the other eigenvalues to both sides of zero; it is at most 0.3 sigma_1^2, so v_1 stays the leading vector whatever the
//        rate was worth, and what ends the iteration is the same: the two agree and stand still.  (One of them alone, until its
//        moves said so, returned v_2 in 1 of 600 slices with sigma_2 = 0.9999 sigma_1 and an rms error of 1.5e-7 instead of
//        1.25e-7 in the timed ones, in 73 us.)  us without and with the shift, noise of 0.5, 1, 2, 3 times the entries of the
//        rank-1 part: m = 64 57 / 50, 67 / 56, 92 / 87, 211 / 212, m = 128 898 / 796, 1150 / 960, 1242 / 1129, 1575 / 1395.  Not
//        at m = 16 and 32, whose slices are one wave that takes as long as its slowest: m = 32 10.5 / 10.5, 13.0 / 12.6, 37 / 37.
//  2. Otherwise (a small gap) H = S^T S is squared and scaled to trace 1 until it has rank 1 - doubling the exponent
//     each time, so the cost grows with the logarithm of 1 / gap and is bounded - and any column of H is v_1.  Orthogonal
//     columns make H diagonal at once.
// Both end in vectors accurate to rounding / gap.
// One warp per slice (four for m = 128), a 4 x 8 grid of lanes, each lane holding an (m/4) x (m/8) patch of S in
// registers for the whole iteration.  A product then needs m/8 (or m/4) values of the vector per lane from shared
// memory and a reduce-scatter over 8 (or 4) lanes; with a whole row per lane every lane would read the whole vector,
// and the 128 bytes per clock that shared memory returns were the limit (149 us for 4096 slices of 64 x 64).
// Bound by fp32 issue: products are packed two to an instruction (fma.rn.f32x2), eight warps share an SM (255 registers).
// Measured, fp32, against the Jacobi iteration: 4096 slices of 64 x 64 with a clear leading value 7714 -> 87 us, Gaussian
// 7690 -> 731 us; 128 x 128 Gaussian 165 -> 18.1 ms; largest error of a Gaussian slice's rank-1 part 2.3e-4 -> 2e-6 (the Jacobi
// iteration stops at a cosine of 2e-6).  Where the columns of a slice are orthogonal up to rounding the squarings run to their
// bound: 0.57 -> 1.29 ms (exactly orthogonal ones of equal length 35 us).
constexpr int kPowerSteps = 40, kPolishSteps = 4, kMaxSquarings = 24;
constexpr float kPowerTol = 1e-6f;
constexpr float kNear = 0.1f, kFast = 0.6f;               // step 1a: distance, and what a step leaves of it

template <int M> struct LeadCfg {
    static constexpr int kWarps = M == 128 ? 4 : 1, kThreads = 32 * kWarps;
    static constexpr int kRows = M / (4 * kWarps), kCols = M / 8;       // a lane's patch of S
    static constexpr int kYC = kRows >= 8 ? kRows / 8 : 1;              // rows of S x a lane ends up with
    static constexpr int kZC = kWarps > 1 || kCols < 4 ? 1 : kCols / 4; // columns of S^T y a thread ends up with
    static constexpr int kPitch = M + 4;                                // of H, floats: rows stay 16-byte aligned
    // the squaring step: kTR x kTC threads, each kRQ x kCQ patches of 4 x 4 of H
    static constexpr int kTC = M <= 16 ? 4 : M == 128 ? 16 : 8, kTR = M == 128 ? 8 : 4;
    static constexpr int kRQ = M / (4 * kTR), kCQ = M / (4 * kTC);
    static constexpr int kSmem = (M * kPitch + 4 * M + (kWarps > 1 ? 2 * kWarps * M : 0)) * (int)sizeof(float);
};

template <int NT> __device__ __forceinline__ void slice_sync()
{
    if (NT == 32) __syncwarp();
    else __syncthreads();
}

// sums over the CTA, the same bits in every thread; `red` has two halves used in turn, so one barrier is enough
template <int NT, int K> __device__ __forceinline__ void slice_sum(float (&v)[K], float (*red)[NT / 32][4], int &phase)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (NT == 32) return;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) red[phase][threadIdx.x >> 5][k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = red[phase][0][k];
#pragma unroll
        for (int w = 1; w < NT / 32; ++w) v[k] += red[phase][w][k];
    }
    phase ^= 1;
}

// Sum v over the lanes that differ in the bits [BIT, BIT_END) of the lane number; afterwards v[0 .. max(1, N >> bits))
// hold this lane's share: the elements from scatter_base(lane) on.
template <int BIT, int BIT_END, int N> __device__ __forceinline__ void reduce_scatter(float *v, int lane)
{
    if constexpr (BIT < BIT_END) {
        if constexpr (N > 1) {
            const bool up = lane >> BIT & 1;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                const float send = up ? v[i] : v[i + N / 2];
                const float keep = up ? v[i + N / 2] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << BIT);
            }
            reduce_scatter<BIT + 1, BIT_END, N / 2>(v, lane);
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1 << BIT);
            reduce_scatter<BIT + 1, BIT_END, 1>(v, lane);
        }
    }
}
template <int BIT, int BIT_END, int N> __device__ __forceinline__ int scatter_base(int lane)
{
    int base = 0, n = N;
#pragma unroll
    for (int b = BIT; b < BIT_END; ++b)
        if (n > 1) {
            n /= 2;
            base += (lane >> b & 1) * n;
        }
    return base;
}

template <int N> __device__ __forceinline__ void load_vec(const float *from, float (&to)[N])
{
    if constexpr (N >= 4) {
#pragma unroll
        for (int i = 0; i < N; i += 4) *reinterpret_cast<float4 *>(to + i) = *reinterpret_cast<const float4 *>(from + i);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) to[i] = from[i];
    }
}

// acc = the calling thread's patches of A^T A, A in shared memory
template <int M>
__device__ __forceinline__ void gram_patches(const float *A, float (&acc)[LeadCfg<M>::kRQ * 4][LeadCfg<M>::kCQ * 4], int tr, int tc)
{
    using C = LeadCfg<M>;
#pragma unroll
    for (int r = 0; r < C::kRQ * 4; ++r)
#pragma unroll
        for (int c = 0; c < C::kCQ * 4; ++c) acc[r][c] = 0.0f;
#pragma unroll 2
    for (int k = 0; k < M; ++k) {
        float a[C::kRQ * 4], b[C::kCQ * 4];
#pragma unroll
        for (int q = 0; q < C::kRQ; ++q)
            *reinterpret_cast<float4 *>(a + 4 * q) = *reinterpret_cast<const float4 *>(A + k * C::kPitch + 4 * (tr + q * C::kTR));
#pragma unroll
        for (int q = 0; q < C::kCQ; ++q)
            *reinterpret_cast<float4 *>(b + 4 * q) = *reinterpret_cast<const float4 *>(A + k * C::kPitch + 4 * (tc + q * C::kTC));
#pragma unroll
        for (int r = 0; r < C::kRQ * 4; ++r)
#pragma unroll
            for (int c = 0; c < C::kCQ * 4; ++c) acc[r][c] = fmaf(a[r], b[c], acc[r][c]);
    }
}

template <typename T, int M>
__global__ void __launch_bounds__(LeadCfg<M>::kThreads)
leading_pair_kernel(const T *__restrict__ A, T *__restrict__ L, T *__restrict__ R)
{
    constexpr bool kShift = M > 32;                          // step 1a
    using C = LeadCfg<M>;
    constexpr int N = M * M, NT = C::kThreads, W = C::kWarps, P = C::kPitch, RH = C::kRows, CW = C::kCols;
    constexpr float kOnce = (float)M / (NT * C::kZC);     // columns are held 1 / kOnce times over the CTA
    static_assert(!kShift || kOnce == 1.0f, "the shift reads elements of x that another thread may have overwritten");
    extern __shared__ __align__(16) float lead_smem[];
    float *H = lead_smem, *x = H + M * P, *y = x + 2 * M; // x[2][M], y[2][M]: the two iterates
    float *part = y + 2 * M;                              // W > 1: [2][W][M] partial sums of S^T y
    __shared__ float red[2][W][4];
    int phase = 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = (warp * 4 + (lane >> 3)) * RH, col0 = (lane & 7) * CW;
    const int my_row = row0 + scatter_base<0, 3, RH>(lane);
    const int my_col = W > 1 ? tid : col0 + scatter_base<3, 5, CW>(lane);
    const int j = blockIdx.x / M, k = blockIdx.x % M;
    const T *slice = A + (size_t)j * N + (size_t)k * M;   // element (l, i) at slice[l * M * N + i]

    f32x2 S[RH][CW / 2];
    auto load_patch = [&](float scale) {
        constexpr int kBytes = CW * (int)sizeof(T), kVec = kBytes < 16 ? kBytes : 16;
        using Vec = typename std::conditional<kVec == 16, uint4, typename std::conditional<kVec == 8, uint2, unsigned>::type>::type;
#pragma unroll
        for (int q = 0; q < RH; ++q) {
            Vec raw[kBytes / kVec];
#pragma unroll
            for (int v = 0; v < kBytes / kVec; ++v)
                raw[v] = reinterpret_cast<const Vec *>(slice + (size_t)(row0 + q) * M * N + col0)[v];
            const T *e = reinterpret_cast<const T *>(raw);
#pragma unroll
            for (int c = 0; c < CW / 2; ++c)
                S[q][c] = pack2(elem<T>::load(e + 2 * c) * scale, elem<T>::load(e + 2 * c + 1) * scale);
        }
    };
    // out = this lane's kYC elements of S v from row my_row on
    auto times_S = [&](const float *v, float (&out)[C::kYC]) {
        float vv[CW], p[RH];
        load_vec(v + col0, vv);
#pragma unroll
        for (int q = 0; q < RH; ++q) {
            f32x2 acc = 0;
#pragma unroll
            for (int c = 0; c < CW / 2; ++c) acc = fma2(S[q][c], pack2(vv[2 * c], vv[2 * c + 1]), acc);
            const float2 t = unpack2(acc);
            p[q] = t.x + t.y;
        }
        reduce_scatter<0, 3, RH>(p, lane);
#pragma unroll
        for (int i = 0; i < C::kYC; ++i) out[i] = p[i];
    };
    // out = this lane's share of S^T v over the rows of its warp
    auto times_St = [&](const float *v, float (&out)[CW]) {
        float vv[RH];
        load_vec(v + row0, vv);
        f32x2 acc[CW / 2];
#pragma unroll
        for (int c = 0; c < CW / 2; ++c) acc[c] = 0;
#pragma unroll
        for (int q = 0; q < RH; ++q)
#pragma unroll
            for (int c = 0; c < CW / 2; ++c) acc[c] = fma2(S[q][c], pack2(vv[q], vv[q]), acc[c]);
#pragma unroll
        for (int c = 0; c < CW / 2; ++c) {
            const float2 t = unpack2(acc[c]);
            out[2 * c] = t.x;
            out[2 * c + 1] = t.y;
        }
        reduce_scatter<3, 5, CW>(out, lane);
    };
    // za = elements my_col .. of S^T ya; BOTH: zb of S^T yb
    auto back = [&](auto both, const float *ya, const float *yb, float (&za)[C::kZC], float (&zb)[C::kZC]) {
        constexpr bool BOTH = decltype(both)::value;
        float a[CW], b[CW];
        times_St(ya, a);
        if (BOTH) times_St(yb, b);
        if constexpr (W > 1) {
            const int at = warp * M + col0 + scatter_base<3, 5, CW>(lane);
#pragma unroll
            for (int i = 0; i < CW / 4; ++i) {
                part[at + i] = a[i];
                if (BOTH) part[W * M + at + i] = b[i];
            }
            __syncthreads();
            za[0] = zb[0] = 0.0f;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                za[0] += part[w * M + tid];
                if (BOTH) zb[0] += part[(W + w) * M + tid];
            }
        } else {
#pragma unroll
            for (int i = 0; i < C::kZC; ++i) {
                za[i] = a[i];
                if (BOTH) zb[i] = b[i];
            }
        }
    };

    load_patch(1.0f);
    float fro2[1] = {0.0f};
#pragma unroll
    for (int q = 0; q < RH; ++q)
#pragma unroll
        for (int c = 0; c < CW / 2; ++c) {
            const float2 t = unpack2(S[q][c]);
            fro2[0] = fmaf(t.x, t.x, fmaf(t.y, t.y, fro2[0]));
        }
    slice_sum<NT>(fro2, red, phase);
    const float fro = sqrtf(fro2[0]);
    if (fro == 0.0f) {                                    // the same value in every thread
        for (int i = tid; i < M; i += NT) {
            elem<T>::store(L + ((size_t)j * M + i) * M + k, 0.0f);
            elem<T>::store(R + ((size_t)k * M + j) * M + i, 0.0f);
        }
        return;
    }
    // scaled to Frobenius norm 1: sigma_1 is then in [1 / sqrt(m), 1] and a few steps need no normalisation
    const float inv_fro = 1.0f / fro;
#pragma unroll
    for (int q = 0; q < RH; ++q)
#pragma unroll
        for (int c = 0; c < CW / 2; ++c) S[q][c] = fma2(S[q][c], pack2(inv_fro, inv_fro), 0);
    for (int i = tid; i < 2 * M; i += NT) {
        unsigned h = (unsigned)(i + 1) * 0x9E3779B1u;     // an integer hash: values in [-1, 1) without structure
        h ^= h >> 15; h *= 0x85EBCA77u; h ^= h >> 13; h *= 0xC2B2AE3Du; h ^= h >> 16;
        x[i] = (float)(int)h * 4.656612873e-10f;
    }
    slice_sync<NT>();

    for (int round = 0; round < 2; ++round) {
        bool done = round == 1;
        float before[C::kZC] = {}, before_b[C::kZC] = {};
        float apart = 4.0f, shift = 0.0f;                 // squared distance of the two at the last test; step 1a
        int every = 3;                                    // tests when step & every == every
        const int steps = round == 0 ? kPowerSteps : kPolishSteps;
#pragma unroll 1
        for (int step = 0; step < steps; ++step) {
            float ya[C::kYC], yb[C::kYC], a[C::kZC], b[C::kZC];
            times_S(x, ya);
            times_S(x + M, yb);
#pragma unroll
            for (int i = 0; i < C::kYC; ++i) {
                y[my_row + i] = ya[i];
                y[M + my_row + i] = yb[i];
            }
            slice_sync<NT>();
            back(std::true_type(), y, y + M, a, b);
            if (kShift)
#pragma unroll
                for (int i = 0; i < C::kZC; ++i) {
                    a[i] = fmaf(-shift, x[my_col + i], a[i]);
                    b[i] = fmaf(-shift, x[M + my_col + i], b[i]);
                }
            if ((step & every) == every || (kShift && step == 1)) {
                float v[3] = {0.0f, 0.0f, 0.0f}, d[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int i = 0; i < C::kZC; ++i) {
                    v[0] = fmaf(a[i], a[i], v[0]);
                    v[1] = fmaf(b[i], b[i], v[1]);
                    v[2] = fmaf(a[i], b[i], v[2]);
                }
                slice_sum<NT>(v, red, phase);
                const float na = rsqrtf(v[0] * kOnce), nb = copysignf(rsqrtf(v[1] * kOnce), v[2]);
#pragma unroll
                for (int i = 0; i < C::kZC; ++i) {
                    a[i] *= na;
                    b[i] *= nb;
                    d[0] = fmaf(a[i] - b[i], a[i] - b[i], d[0]);
                    d[1] = fmaf(a[i] - before[i], a[i] - before[i], d[1]);
                    d[2] = fmaf(b[i] - before_b[i], b[i] - before_b[i], d[2]);
                    before[i] = a[i];
                    before_b[i] = b[i];
                }
                slice_sum<NT>(d, red, phase);
                constexpr float kSame = kPowerTol * kPowerTol / kOnce;
                const float still = kShift && (every == 1 || step == 3) ? 0.25f * kSame : kSame;      // two steps or four since the last test
                if (kShift && step == 1) {
                    apart = d[0];
                } else if (!(d[1] >= still) && !(d[0] >= kSame)) {
                    done = true;                          // (NaN: nothing to wait for)
                } else if (d[1] < still && d[2] < still) {
                    // both stand still and differ: eigenvectors, of the same singular value or not; the one with the larger is kept
                    done = true;
                    if (v[1] > v[0])
#pragma unroll
                        for (int i = 0; i < C::kZC; ++i) a[i] = b[i];
                } else if (kShift && step == 3 && round == 0 && d[0] * kOnce < kNear * kNear && d[0] < kFast * kFast * kFast * kFast * apart) {
                    shift = 0.5f * sqrtf(sqrtf(v[0] * kOnce * (d[0] / apart)));
                    every = 1;
                }
            }
#pragma unroll
            for (int i = 0; i < C::kZC; ++i) {
                x[my_col + i] = a[i];
                x[M + my_col + i] = b[i];
            }
            slice_sync<NT>();
            if (done && (step & every) == every) break;
        }
        if (done) break;

#pragma unroll
        for (int q = 0; q < RH; ++q)
#pragma unroll
            for (int c = 0; c < CW / 2; ++c) *reinterpret_cast<f32x2 *>(H + (row0 + q) * P + col0 + 2 * c) = S[q][c];
        slice_sync<NT>();
        const int tr = tid / C::kTC, tc = tid % C::kTC;
        const bool on = tr < C::kTR;
        float acc[C::kRQ * 4][C::kCQ * 4];
        bool last = false;
#pragma unroll 1
        for (int sq = 0; sq <= kMaxSquarings; ++sq) {     // pass 0 forms S^T S, the others square it
            gram_patches<M>(H, acc, on ? tr : 0, tc);
            float trace[1] = {0.0f};
            if (on)
#pragma unroll
                for (int r = 0; r < C::kRQ * 4; ++r)
#pragma unroll
                    for (int c = 0; c < C::kCQ * 4; ++c)
                        if (4 * (tr + r / 4 * C::kTR) + r % 4 == 4 * (tc + c / 4 * C::kTC) + c % 4) trace[0] += acc[r][c];
            if (sq == 0) {                                // all products of different columns zero: the longest column is the answer
                float off[1] = {0.0f};
                if (on)
#pragma unroll
                    for (int r = 0; r < C::kRQ * 4; ++r)
#pragma unroll
                        for (int c = 0; c < C::kCQ * 4; ++c)
                            if (4 * (tr + r / 4 * C::kTR) + r % 4 != 4 * (tc + c / 4 * C::kTC) + c % 4 && acc[r][c] != 0.0f) off[0] = 1.0f;
                slice_sum<NT>(off, red, phase);
                last = off[0] == 0.0f;
            }
            slice_sum<NT>(trace, red, phase);
            slice_sync<NT>();                             // the reads of H are over
            const float scale = 1.0f / trace[0];
            if (on)
#pragma unroll
                for (int r = 0; r < C::kRQ * 4; ++r)
#pragma unroll
                    for (int c = 0; c < C::kCQ * 4; c += 4)
                        *reinterpret_cast<float4 *>(H + (4 * (tr + r / 4 * C::kTR) + r % 4) * P + 4 * (tc + c / 4 * C::kTC)) =
                            make_float4(acc[r][c] * scale, acc[r][c + 1] * scale, acc[r][c + 2] * scale, acc[r][c + 3] * scale);
            slice_sync<NT>();
            if (last) break;
            // trace 1 before squaring: 1 - trace(H^2) is about 2 (lambda_2 / lambda_1)^(2^sq); the next squaring squares it
            last = sq > 0 && 1.0f - trace[0] < 1e-3f;
        }
        float best = -1.0f;
        int at = 0;
        for (int i = 0; i < M; ++i) {
            const float d = H[i * P + i];
            if (d > best) { best = d; at = i; }
        }
        for (int i = tid; i < M; i += NT) x[i] = x[M + i] = H[at * P + i];
        load_patch(inv_fro);
        slice_sync<NT>();
    }

    float u[C::kYC], z[C::kZC], unused[C::kZC];
    times_S(x, u);
    float s2[1] = {0.0f};
#pragma unroll
    for (int i = 0; i < C::kYC; ++i) s2[0] = fmaf(u[i], u[i], s2[0]);
    slice_sum<NT>(s2, red, phase);
    s2[0] *= (float)M / (NT * C::kYC);
    const float inv_sigma = rsqrtf(s2[0]), root = sqrtf(fro * sqrtf(s2[0]));
#pragma unroll
    for (int i = 0; i < C::kYC; ++i) {
        u[i] *= inv_sigma;
        y[my_row + i] = u[i];
        elem<T>::store(L + ((size_t)j * M + my_row + i) * M + k, root * u[i]);
    }
    slice_sync<NT>();
    back(std::false_type(), y, nullptr, z, unused);       // sigma_1 v_1 of the scaled slice
#pragma unroll
    for (int i = 0; i < C::kZC; ++i)
        elem<T>::store(R + ((size_t)k * M + j) * M + my_col + i, fro / root * z[i]);
}

template <typename T, int M>
int launch_leading_pair(const void *A, void *L, void *R, cudaStream_t s)
{
    auto kern = leading_pair_kernel<T, M>;
    constexpr int smem = LeadCfg<M>::kSmem;
    if (smem > 48 * 1024) MONARCH_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    kern<<<M * M, LeadCfg<M>::kThreads, smem, s>>>((const T *)A, (T *)L, (T *)R);
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

template <typename T, int M>
int launch_project(const void *A, void *L, void *R, unsigned long long *rotations, cudaStream_t s)
{
    return rotations != nullptr ? launch_jacobi<T, M>(A, L, R, rotations, s) : launch_leading_pair<T, M>(A, L, R, s);
}

template <typename T>
int project_t(const void *A, void *L, void *R, int m, unsigned long long *rotations, cudaStream_t s)
{
    switch (m) {
        case 16:  return launch_project<T, 16>(A, L, R, rotations, s);
        case 32:  return launch_project<T, 32>(A, L, R, rotations, s);
        case 64:  return launch_project<T, 64>(A, L, R, rotations, s);
        case 128: return launch_project<T, 128>(A, L, R, rotations, s);
    }
    return MONARCH_ERR_UNSUPPORTED;
}

}  // namespace

int dense_from_factors(const void *L, const void *R, void *M, int m, int dtype, cudaStream_t s)
{
    const int n = m * m, per = kDenseVecs * 256 * (dtype == MONARCH_F32 ? 4 : 8);
    const dim3 grid((unsigned)m, (unsigned)(m / kDenseRows), (unsigned)((n + per - 1) / per));
    if (dtype == MONARCH_F32)
        dense_kernel<float><<<grid, 256, 0, s>>>((const float *)L, (const float *)R, (float *)M, m);
    else
        dense_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>((const __nv_bfloat16 *)L, (const __nv_bfloat16 *)R,
                                                         (__nv_bfloat16 *)M, m);
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

int project_to_factors(const void *A, void *L, void *R, int m, int dtype, unsigned long long *rotations, cudaStream_t s)
{
    return dtype == MONARCH_F32 ? project_t<float>(A, L, R, m, rotations, s)
                                : project_t<__nv_bfloat16>(A, L, R, m, rotations, s);
}

}  // namespace monarch
