// Forward y = P L P^T R x for m = 16 (n = 256) in one launch on the CUDA cores, fp32 or bf16 storage with fp32
// arithmetic.  A token vector is 256 elements, so a CTA keeps a few tokens and their intermediate u' in shared
// memory and runs both stages of Section 3.3 (steps 1-3) back to back: thread e = j*16 + k forms
// u'[t][j][k] = sum_i R[k][j][i] x[t][k*16+i] with its row of R in registers, then thread e = l*16 + j forms
// y[t][l*16+j] = sum_k L[j][l][k] u'[t][j][k].  At this size the two-launch chain is bound by launch latency;
// one launch halves it.  (Blocks of 16 x 16 are below the tensor-core tile: fp32 FMA is the right unit, and in
// fp32 mode the only one that meets the 1e-5 tolerance.)
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

template <typename T>
int launch_m16(const void *x, const void *L, const void *R, void *y, int64_t tokens, cudaStream_t s)
{
    if (tokens == 0) return MONARCH_OK;
    // One token per CTA while every CTA has an SM of its own; then as many tokens per CTA as it takes.  Beyond a few
    // hundred tokens the automatic choice is another family.
    auto run = [&](auto kern, int per) {
        kern<<<(unsigned)((tokens + per - 1) / per), kN16, 0, s>>>((const T *)x, (const T *)L, (const T *)R, (T *)y, tokens);
    };
    if (tokens <= 148) run(fused_fwd_m16_kernel<T, 1>, 1);
    else if (tokens <= 296) run(fused_fwd_m16_kernel<T, 2>, 2);
    else run(fused_fwd_m16_kernel<T, 8>, 8);
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
