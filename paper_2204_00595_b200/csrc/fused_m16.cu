// Forward y = P L P^T R x for m = 16 (n = 256) in one launch on the CUDA cores, fp32 or bf16 storage with fp32
// arithmetic.  A token vector is 256 elements, so a CTA keeps a few tokens and their intermediate u' in shared
// memory and runs both stages of Section 3.3 (steps 1-3) back to back: thread e = j*16 + k forms
// u'[t][j][k] = sum_i R[k][j][i] x[t][k*16+i] with its row of R in registers, then thread e = l*16 + j forms
// y[t][l*16+j] = sum_k L[j][l][k] u'[t][j][k].  At this size the two-launch chain is bound by launch latency;
// one launch halves it.  fp32 multiply-adds in both dtypes: u' is never rounded.
#include "common.cuh"

namespace monarch {
namespace {

constexpr int kM16 = 16, kN16 = 256;

// 16 consecutive elements as 16-byte loads
template <typename T> __device__ __forceinline__ void load_row(const T *p, float (&w)[kM16])
{
    constexpr int V = 16 / sizeof(T);
    uint4 raw[kM16 / V];
#pragma unroll
    for (int q = 0; q < kM16 / V; ++q) raw[q] = reinterpret_cast<const uint4 *>(p)[q];
#pragma unroll
    for (int i = 0; i < kM16; ++i) w[i] = elem<T>::load(reinterpret_cast<const T *>(raw) + i);
}

// Bound by latency: one trip to memory (inputs and both rows of weights are requested together, the rows 16 bytes at a
// time), two short products with a barrier between them, one store.
template <typename T, int TOK>
__global__ void __launch_bounds__(kN16) fused_fwd_m16_kernel(const T *__restrict__ x, const T *__restrict__ L,
                                                             const T *__restrict__ R, T *__restrict__ y,
                                                             long long tokens)
{
    __shared__ __align__(16) float xs[TOK][kN16];
    __shared__ __align__(16) float us[TOK][kN16];
    const int e = threadIdx.x;
    const long long t0 = (long long)blockIdx.x * TOK;
    const int left = (int)(tokens - t0 < TOK ? tokens - t0 : TOK);
    const int hi = e >> 4, lo = e & 15;                // stage 1: j = hi, k = lo; stage 2: l = hi, j = lo
    float wl[kM16], wr[kM16], in[TOK];
#pragma unroll
    for (int t = 0; t < TOK; ++t) in[t] = t < left ? elem<T>::load(x + (t0 + t) * kN16 + e) : 0.0f;
    load_row(R + (lo * kM16 + hi) * kM16, wr);
    load_row(L + (lo * kM16 + hi) * kM16, wl);
#pragma unroll
    for (int t = 0; t < TOK; ++t) xs[t][e] = in[t];
    __syncthreads();
    auto times = [&](const float (&w)[kM16], const float *v) {
        float acc = 0.0f;
#pragma unroll
        for (int i = 0; i < kM16; i += 4) {
            const float4 q = *reinterpret_cast<const float4 *>(v + i);
            acc = fmaf(w[i], q.x, acc);
            acc = fmaf(w[i + 1], q.y, acc);
            acc = fmaf(w[i + 2], q.z, acc);
            acc = fmaf(w[i + 3], q.w, acc);
        }
        return acc;
    };
    // u'[j][k] = sum_i R[k][j][i] x[k*16 + i], kept at [j*16 + k]
#pragma unroll
    for (int t = 0; t < TOK; ++t) us[t][e] = times(wr, xs[t] + lo * kM16);
    __syncthreads();
    // y[l*16 + j] = sum_k L[j][l][k] u'[j][k]
#pragma unroll
    for (int t = 0; t < TOK; ++t)
        if (t < left) elem<T>::store(y + (t0 + t) * kN16 + e, times(wl, us[t] + lo * kM16));
}

// ---- many tokens
// 64 threads and four tokens at a time.  Stage 1: a thread has block k of R and rows j = g, g + 4, g + 8, g + 12 of it, stage 2
// block j of L and rows l likewise, as fp32 pairs of rows in registers (fma.rn.f32x2; every sum runs over its 16 terms in order, so
// the bits are those of the kernel above).  u' stays fp32 in shared memory: as tensor-core operands it would have to be rounded to
// bf16, which makes the error of y 1.41 times as large.  x and u' lie as [token][block][four pieces of 4], the pieces permuted so
// that the eight blocks of a warp fall on different banks.  Bound by fp32 issue: 8192 multiply-adds per token, 7.4 us of the
// chip's rate at 32768 tokens.  Measured there, bf16: 20.6 us (the units with u' rounded 24.7, eight tokens per CTA with the weights
// read by each 213), 1000 tokens 4.6.
constexpr int kGroup = 4, kRowThreads = 64;

__device__ __forceinline__ int piece_at(int block, int c)         // of four floats
{
    return block * 4 + (c ^ ((block & 2) | (block >> 2 & 1)));
}

// Rows r0, r0 + 4, r0 + 8, r0 + 12 of one block: two pairs for each of the 16 columns
template <typename T> __device__ __forceinline__ void load_pairs(const T *block, int r0, f32x2 (&w)[2][kM16])
{
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        float a[kM16], b[kM16];
        load_row(block + (r0 + 8 * p) * kM16, a);
        load_row(block + (r0 + 8 * p + 4) * kM16, b);
#pragma unroll
        for (int i = 0; i < kM16; ++i) w[p][i] = pack2(a[i], b[i]);
    }
}

// acc[t][p] = the sums of pair p for token t, inputs of one block
__device__ __forceinline__ void times_pairs(const f32x2 (&w)[2][kM16], const float4 (*in)[kN16 / 4], int block, f32x2 (&acc)[kGroup][2])
{
#pragma unroll
    for (int t = 0; t < kGroup; ++t) acc[t][0] = acc[t][1] = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int t = 0; t < kGroup; ++t) {
            const float4 v = in[t][piece_at(block, c)];
            const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f32x2 d = pack2(e[i], e[i]);
                acc[t][0] = fma2(w[0][c * 4 + i], d, acc[t][0]);
                acc[t][1] = fma2(w[1][c * 4 + i], d, acc[t][1]);
            }
        }
}

template <typename T>
__global__ void __launch_bounds__(kRowThreads, 4) rows_fwd_m16_kernel(const T *__restrict__ x, const T *__restrict__ L,
                                                                      const T *__restrict__ R, T *__restrict__ y, long long tokens)
{
    constexpr int V = 16 / (int)sizeof(T), kVecs = kGroup * kN16 / V / kRowThreads, kRow = kN16 / V;   // 16-byte accesses
    __shared__ float4 xs[kGroup][kN16 / 4], us[kGroup][kN16 / 4];
    __shared__ __align__(16) T ys[kGroup][kN16];
    const int tid = threadIdx.x, b = (tid >> 5) * 8 + (tid & 7), g = tid >> 3 & 3;
    const long long groups = (tokens + kGroup - 1) / kGroup;
    uint4 raw[kVecs];
    auto fetch = [&](long long group) {
#pragma unroll
        for (int q = 0; q < kVecs; ++q) {
            const int v = q * kRowThreads + tid;
            const long long t = group * kGroup + v / kRow;
            raw[q] = t < tokens ? reinterpret_cast<const uint4 *>(x + t * kN16)[v % kRow] : make_uint4(0, 0, 0, 0);
        }
    };
    auto send = [&](long long group) {
#pragma unroll
        for (int q = 0; q < kVecs; ++q) {
            const int v = q * kRowThreads + tid;
            const long long t = group * kGroup + v / kRow;
            if (t < tokens) reinterpret_cast<uint4 *>(y + t * kN16)[v % kRow] = reinterpret_cast<const uint4 *>(ys[v / kRow])[v % kRow];
        }
    };
    fetch(blockIdx.x);
    f32x2 wr[2][kM16], wl[2][kM16];
    load_pairs(R + b * kM16 * kM16, g, wr);
    load_pairs(L + b * kM16 * kM16, g, wl);
    long long last = -1;
    for (long long group = blockIdx.x; group < groups; group += gridDim.x) {
#pragma unroll
        for (int q = 0; q < kVecs; ++q) {
            const int v = q * kRowThreads + tid, first = v % kRow * V;      // column
            const T *e = reinterpret_cast<const T *>(&raw[q]);
#pragma unroll
            for (int h = 0; h < V; h += 4)
                xs[v / kRow][piece_at(first / kM16, (first % kM16 + h) / 4)] =
                    make_float4(elem<T>::load(e + h), elem<T>::load(e + h + 1), elem<T>::load(e + h + 2), elem<T>::load(e + h + 3));
        }
        if (group + gridDim.x < groups) fetch(group + gridDim.x);
        __syncthreads();                                   // x is here, the last y is complete
        if (last >= 0) send(last);
        f32x2 acc[kGroup][2];
        times_pairs(wr, xs, b, acc);
#pragma unroll
        for (int t = 0; t < kGroup; ++t)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const float2 u = unpack2(acc[t][p]);       // rows j = g + 8 p and g + 8 p + 4 of block k = b
                float *row = reinterpret_cast<float *>(us[t]);
                row[piece_at(g + 8 * p, b >> 2) * 4 + (b & 3)] = u.x;
                row[piece_at(g + 8 * p + 4, b >> 2) * 4 + (b & 3)] = u.y;
            }
        __syncthreads();                                   // u' is complete, x and the last y have been read
        times_pairs(wl, us, b, acc);
#pragma unroll
        for (int t = 0; t < kGroup; ++t)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const float2 v = unpack2(acc[t][p]);
                elem<T>::store(&ys[t][(g + 8 * p) * kM16 + b], v.x);
                elem<T>::store(&ys[t][(g + 8 * p + 4) * kM16 + b], v.y);
            }
        last = group;
    }
    __syncthreads();
    if (last >= 0) send(last);
}

template <typename T>
int launch_m16(const void *x, const void *L, const void *R, void *y, int64_t tokens, cudaStream_t s)
{
    if (tokens == 0) return MONARCH_OK;
    auto run = [&](auto kern, int threads, long long ctas) {
        kern<<<(unsigned)ctas, threads, 0, s>>>((const T *)x, (const T *)L, (const T *)R, (T *)y, tokens);
    };
    // one token per CTA while every CTA has an SM of its own, then two; beyond, four CTAs per SM walk over the tokens
    if (tokens <= 148) run(fused_fwd_m16_kernel<T, 1>, kN16, tokens);
    else if (tokens <= 256) run(fused_fwd_m16_kernel<T, 2>, kN16, (tokens + 1) / 2);
    else {
        int sms = 0;
        MONARCH_TRY(current_device_sms(&sms));
        const long long groups = (tokens + kGroup - 1) / kGroup, most = 4LL * sms;
        run(rows_fwd_m16_kernel<T>, kRowThreads, groups < most ? groups : most);
    }
    note_launch();
    MONARCH_CUDA_TRY(cudaGetLastError());
    return MONARCH_OK;
}

}  // namespace

int fused_fwd_m16(const void *x, const void *L, const void *R, void *y, int64_t tokens, int dtype, cudaStream_t s)
{
    return dtype == MONARCH_F32 ? launch_m16<float>(x, L, R, y, tokens, s)
                                : launch_m16<__nv_bfloat16>(x, L, R, y, tokens, s);
}

}  // namespace monarch
