// Shared host/device helpers of libmonarch (internal; not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "monarch.h"

namespace monarch {

// Launch counter behind monarch_launch_count().
void note_launch(int n = 1);

// SM count of the current device (cached per device ordinal, safe against concurrent first calls).
int current_device_sms(int *sms);

// A value cached per device ordinal (an occupancy figure): get() returns -1 until set() has stored one for the current
// device.  Two threads racing on a first call both compute and store the same value.
struct PerDeviceCache {
    std::atomic<int> v[64];                  // value + 1; zero-initialised as a static
    int get() const
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
        return v[dev].load(std::memory_order_relaxed) - 1;
    }
    void set(int value)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) v[dev].store(value + 1, std::memory_order_relaxed);
    }
};

#define MONARCH_CUDA_TRY(expr)                                   \
    do {                                                         \
        cudaError_t err_ = (expr);                               \
        if (err_ != cudaSuccess) return MONARCH_ERR_CUDA;        \
    } while (0)

#define MONARCH_TRY(expr)                                        \
    do {                                                         \
        int st_ = (expr);                                        \
        if (st_ != MONARCH_OK) return st_;                       \
    } while (0)

template <typename T> struct elem;
template <> struct elem<float> {
    static __device__ __forceinline__ float load(const float *p) { return *p; }
    static __device__ __forceinline__ void store(float *p, float v) { *p = v; }
};
template <> struct elem<__nv_bfloat16> {
    static __device__ __forceinline__ float load(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// Two fp32 values in a register pair; fma2 rounds each half like fmaf, in one instruction for both.
typedef unsigned long long f32x2;
static __device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
static __device__ __forceinline__ f32x2 pack2(float x, float y)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
static __device__ __forceinline__ float2 unpack2(f32x2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}

// erf form of GELU, evaluated in fp32.
static __device__ __forceinline__ float gelu_erf(float a)
{
    return 0.5f * a * (1.0f + erff(a * 0.70710678118654752440f));
}

// d/da of a/2 (1 + erf(a / sqrt 2)):  Phi(a) + a phi(a)
static __device__ __forceinline__ float gelu_erf_grad(float a)
{
    const float cdf = 0.5f * (1.0f + erff(a * 0.70710678118654752440f));
    return cdf + a * 0.39894228040143267794f * expf(-0.5f * a * a);
}

// GELU(a) = a/2 (1 + erf(a / sqrt 2)) evaluated as a * sigmoid(2 a (c0 + c1 a^2 + c2 a^4)): the logistic form
// of the usual tanh approximation with one more polynomial term, coefficients fitted (minimax over [-8, 8]) to
// the erf definition: |error| <= 2.6e-5 everywhere (a^2 is clamped at 64, beyond which the sigmoid has
// saturated) - well below one bf16 ulp of the result.  Nine instructions, two of them MUFU; the libm-grade erf
// costs twice that.  Used where the result is rounded to bf16 anyway; fp32 paths use gelu_erf.
static __device__ __forceinline__ float gelu_fast_exp(float a)               // exp(-2 a poly(a^2))
{
    const float a2 = fminf(a * a, 64.0f);
    float t = fmaf(a2, 0.0010142630198970437f, -0.10677572339773178f);     // -2 log2(e) * (c2 a^2 + c1)
    t = fmaf(a2, t, -2.301121234893799f);
    // flush-to-zero forms: no range fix-up code around the two MUFU operations (the exponent is at most 40 for
    // |a| <= 8; beyond that 2^x overflows to inf or flushes to 0 and the sigmoid saturates to 0 or 1, as it should)
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(a * t));
    return e;
}
static __device__ __forceinline__ float gelu_fast(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + gelu_fast_exp(a)));
    return a * r;
}

// The same for two values, bit for bit, with packed instructions where there are any: 12 to issue instead of 18 (block of 4000
// tokens at m = 128: 247 -> 241 us; m = 32, 16000 tokens: 40.6 -> 40.0; m = 64, where the GELU stands between the products of the
// middle launch, 32768 tokens: 391 -> 381).  One reciprocal for both, of the product of their denominators, takes more
// instructions: nothing gained at m = 64 (391), 18 % lost at m = 128.
static __device__ __forceinline__ void gelu_fast2(float &a, float &b)
{
    asm("{\n\t"
        ".reg .b64 x, q, t, c;\n\t"
        ".reg .f32 u, v, one;\n\t"
        "mov.b64 x, {%0, %1};\n\t"
        "mul.rn.f32x2 q, x, x;\n\t"
        "mov.b64 {u, v}, q;\n\t"
        "min.f32 u, u, 0f42800000;\n\t"
        "min.f32 v, v, 0f42800000;\n\t"
        "mov.b64 q, {u, v};\n\t"
        "mov.b64 t, {%2, %2};\n\t"
        "mov.b64 c, {%3, %3};\n\t"
        "fma.rn.f32x2 t, q, t, c;\n\t"
        "mov.b64 c, {%4, %4};\n\t"
        "fma.rn.f32x2 t, q, t, c;\n\t"
        "mul.rn.f32x2 t, x, t;\n\t"
        "mov.b64 {u, v}, t;\n\t"
        "ex2.approx.ftz.f32 u, u;\n\t"
        "ex2.approx.ftz.f32 v, v;\n\t"
        "mov.b64 t, {u, v};\n\t"
        "mov.f32 one, 0f3F800000;\n\t"
        "mov.b64 c, {one, one};\n\t"
        "add.rn.f32x2 t, t, c;\n\t"
        "mov.b64 {u, v}, t;\n\t"
        "rcp.approx.ftz.f32 u, u;\n\t"
        "rcp.approx.ftz.f32 v, v;\n\t"
        "mov.b64 t, {u, v};\n\t"
        "mul.rn.f32x2 t, x, t;\n\t"
        "mov.b64 {%0, %1}, t;\n\t"
        "}"
        : "+f"(a), "+f"(b)
        : "f"(0.0010142630198970437f), "f"(-0.10677572339773178f), "f"(-2.301121234893799f));
}

// d/da GELU(a) = Phi(a) + a phi(a) with Phi from the same sigmoid (|Phi error| <= 5.1e-5) and the normal
// density phi evaluated directly: |error| <= 5.1e-5, for results that are rounded to bf16.
static __device__ __forceinline__ float gelu_fast_grad(float a)
{
    const float pdf = 0.39894228040143267794f * exp2f(-0.72134752044448170368f * a * a);
    return fmaf(a, pdf, __fdividef(1.0f, 1.0f + gelu_fast_exp(a)));
}

// ---- staged (one block-diagonal stage per launch) kernels, staged_simt.cu ----
// Workspace layout helpers and launchers; every launcher returns a monarch_status_t.
size_t staged_workspace_bytes(int op, int64_t tokens, int32_t n, int32_t m, int dtype);
int staged_fwd(const void *x, const void *L, const void *R, void *y, int64_t tokens, int m,
               int dtype, void *ws, cudaStream_t s);
int staged_bwd_dx(const void *dy, const void *L, const void *R, void *dx, int64_t tokens, int m,
                  int dtype, void *ws, cudaStream_t s);
int staged_bwd_dw(const void *x, const void *dy, const void *L, const void *R, float *dL,
                  float *dR, int accumulate, int64_t tokens, int m, int dtype, void *ws,
                  cudaStream_t s);
int staged_mlp_fwd(const void *x, const void *L1, const void *R1, const void *b1, const void *L2,
                   const void *R2, const void *b2, void *y, int64_t tokens, int m, int dtype,
                   void *ws, cudaStream_t s);


// ---- the feed-forward block at m = 128 as four launches of a tensor-core stage (tc_stage.cu): where the forward of
// chain_m128.cu cannot run as one launch ----
int tc_staged_mlp_fwd(const void *x, const void *L1, const void *R1, const void *b1, const void *L2,
                      const void *R2, const void *b2, void *y, int64_t tokens, void *ws, cudaStream_t s);


// m = 128 as chains of block GEMMs on token-innermost planes (chain_m128.cu)
size_t chain_fwd_m128_workspace_bytes(int64_t tokens);
size_t chain_bwd_m128_workspace_bytes(int64_t tokens);
int chain_fwd_m128(const void *x, const void *L, const void *R, void *y, int64_t tokens, void *ws, cudaStream_t s);
// y = M2 GELU(M1 x + b1) + b2 in two launches; workspace 0 where the one-launch forward cannot run
size_t chain_mlp_fwd_m128_workspace_bytes(int64_t tokens);
int chain_mlp_fwd_m128(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2,
                       void *y, int64_t tokens, void *ws, cudaStream_t s);
// saved_up: the u' the forward call left in its workspace (chain_fwd_m128_saved_u), or null
int chain_bwd_m128(const void *x, const void *dy, const void *L, const void *R, const void *saved_up, void *dx, float *dL,
                   float *dR, int accumulate, int want_dx, int want_dw, int64_t tokens, void *ws, cudaStream_t s);
const void *chain_fwd_m128_saved_u(const void *fwd_ws, int64_t tokens);
// test aid: the next plane-transpose launch (last step of the m = 128 forward) leaves out the load of this item
void debug_skip_next_plane_load(long long item);
// test aid: the item that the first launch of the next m = 32 or m = 64 call leaves out, once; -1: none
int take_skipped_tile();
// true when the next forward call has to run as three launches: the switch for comparison runs, or a load to leave out
bool chain_fwd_m128_split();

// ---- forward for m = 16 in one launch on the CUDA cores, both dtypes (fused_m16.cu); no workspace use ----
int fused_fwd_m16(const void *x, const void *L, const void *R, void *y, int64_t tokens, int dtype, cudaStream_t s);

// ---- m = 32, bf16: all stages of a token tile inside one CTA (fused_m32.cu) ----
// forward: workspace = status word only
int fused_fwd_m32(const void *x, const void *L, const void *R, void *y, int64_t tokens, void *ws, cudaStream_t s);
// the feed-forward block in two launches
size_t fused_mlp_fwd_m32_workspace_bytes(int64_t tokens);
int fused_mlp_fwd_m32(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2,
                      void *y, int64_t tokens, void *ws, cudaStream_t s);
// dx null: gradients only; dL null: dx only.  The gradients are sums in a fixed order.
// Reported on top while monarch_set_deterministic is on, as its contract says (these kernels have no use for it).
constexpr size_t kTcPartialBytes = (size_t)32 << 20;
size_t fused_bwd_m32_workspace_bytes(int64_t tokens);
int fused_bwd_m32(const void *x, const void *dy, const void *L, const void *R, void *dx, float *dL, float *dR, int accumulate,
                  int64_t tokens, void *ws, cudaStream_t s);

// ---- m = 64, bf16: one streaming launch per stage (stream_m64.cu) ----
size_t fused_fwd_m64_workspace_bytes(int64_t tokens);
int fused_fwd_m64(const void *x, const void *L, const void *R, void *y, int64_t tokens, void *ws, cudaStream_t s);
// where the forward keeps u inside its workspace
const void *fused_fwd_m64_saved_u(const void *fwd_ws);
// one pass y = M x + bias; workspace of fused_fwd_m64 (u stays behind)
int fused_fwd_bias_m64(const void *x, const void *L, const void *R, const void *bias, void *y, int64_t tokens, void *ws, void *status,
                       cudaStream_t s);
size_t fused_mlp_fwd_m64_workspace_bytes(int64_t tokens);
int fused_mlp_fwd_m64(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2, void *y,
                      int64_t tokens, void *ws, cudaStream_t s);
int fused_cplx_m64(const void *x, const void *L, const void *R, void *y, int adjoint, int64_t tokens, void *ws, cudaStream_t s);
size_t fused_bwd_dx_m64_workspace_bytes(int64_t tokens);
int fused_bwd_dx_m64(const void *dy, const void *L, const void *R, void *dx, int64_t tokens, void *ws, cudaStream_t s);
// dx null: gradients only.  u_saved null: recomputed.  The gradients are sums in a fixed order.
size_t fused_bwd_m64_workspace_bytes(int64_t tokens);
int fused_bwd_m64(const void *x, const void *dy, const void *L, const void *R, const void *u_saved, void *dx, float *dL, float *dR,
                  int accumulate, int64_t tokens, void *ws, cudaStream_t s);

// ---- general (rectangular) Monarch multiply on the CUDA cores (rect_simt.cu); workspace = [status][u] ----
size_t rect_workspace_bytes(int64_t tokens, int q, int b, int dtype);
// wt = 1 reads the blocks transposed (the adjoint passes of the backward call)
int rect_stage1_simt(const void *x, const void *R, void *u, int64_t tokens, int q, int b1, int b, int dtype, int wt,
                     cudaStream_t s);
int rect_stage2_simt(const void *u, const void *Lp, void *y, int64_t tokens, int q, int b, int r, int dtype, int wt,
                     cudaStream_t s);
// want_dL / want_dR = 0: that gradient comes from the streaming pass / the tensor-core kernel
int rect_wgrad_simt(const void *x, const void *dy, const void *u, const void *du, float *dL, float *dR, int64_t tokens,
                    int q, int b1, int b, int r, int dtype, int want_dL, int want_dR, cudaStream_t s);
// stage 1 on the tensor cores (rect_tc.cu): bf16, b1 and b multiples of 64
bool rect_stage1_tc_available(int q, int b1, int b, int dtype);
int rect_stage1_tc(const void *x, const void *R, void *u, int64_t tokens, int q, int b1, int b, unsigned *status,
                   cudaStream_t s);
int rect_stage1_adjoint_tc(const void *du, const void *R, void *dx, int64_t tokens, int q, int b1, int b,
                           unsigned *status, cudaStream_t s);
// du = L^T dy and dL += for blocks up to 4 x 4 in one TMA-fed streaming pass (rect_tc.cu): sizes as rect_stage2_stream_available;
// zero[0 .. zero_n) is zeroed beside
int rect_bwd_stream(const void *dy, const void *u, const void *Lp, void *du, float *dL, int64_t tokens, int q, int b, int r,
                    unsigned *status, float *zero, size_t zero_n, cudaStream_t s);
bool rect_wgrad_R_tc_available(int q, int b1, int b, int dtype);
// dR (+)= ...: _adds says whether the sums are added to what is in dR, so that the caller zeroes it first unless it accumulates
int rect_wgrad_R_tc_adds(int64_t tokens, int q, int b1, int b, bool *adds);
int rect_wgrad_R_tc(const void *du, const void *x, float *dR, int accumulate, int64_t tokens, int q, int b1, int b, unsigned *status,
                    cudaStream_t s);
// stage 2 as a TMA-fed streaming pass (rect_tc.cu): bf16, q and r at most 4, b a multiple of 8 and at least 128
bool rect_stage2_stream_available(int q, int b, int r, int dtype);
int rect_stage2_stream(const void *u, const void *Lp, void *y, int64_t tokens, int q, int b, int r, unsigned *status, cudaStream_t s);

// ---- rectangular class with wrapped-diagonal blocks, b2 != b3 (rect_wrapped.cu) ----
size_t rectw_workspace_bytes(int64_t tokens, int q, int b2, int b3, int r, int dtype);
size_t rectw_bwd_workspace_bytes(int64_t tokens, int q, int b2, int b3, int r, int dtype);
int rectw_fwd(const void *x, const void *Lw, const void *R, void *y, int64_t tokens, int q, int b1, int b2, int b3, int r,
              int dtype, bool fast, void *ws, cudaStream_t s);
int rectw_bwd(const void *x, const void *dy, const void *Lw, const void *R, void *dx, float *dLw, float *dR, int accumulate,
              int64_t tokens, int q, int b1, int b2, int b3, int r, int dtype, bool fast, void *ws, cudaStream_t s);

// ---- whole calls as one cooperative launch over units of block products, both dtypes, any m (block_units.cu) ----
// u, u_saved: the intermediate of the forward call in this family's own layout
namespace units {
// where a forward call leaves u in its workspace: after the status area and the counters of the other kernels, which
// have to stay zero
void *saved_u(const void *fwd_ws);
size_t workspace_bytes(int op, int64_t tokens, int m, int dtype);
int fwd(const void *x, const void *L, const void *R, void *y, int64_t tokens, int m, int dtype, void *u, void *ws, cudaStream_t s);
// dx null: weight gradients only; dL null: dx only; u_saved null: recomputed
int bwd(const void *x, const void *dy, const void *L, const void *R, const void *u_saved, void *dx, float *dL, float *dR,
        int accumulate, int64_t tokens, int m, int dtype, void *ws, cudaStream_t s);
int mlp_fwd(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2, void *y,
            int64_t tokens, int m, int dtype, void *ws, cudaStream_t s);
int mlp_bwd(const void *x, const void *dy, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, void *dx,
            float *dL1, float *dR1, float *db1, float *dL2, float *dR2, float *db2, int accumulate, int64_t tokens, int m, int dtype,
            void *ws, cudaStream_t s);
}  // namespace units

// ---- dense <-> Monarch factors (project.cu): Eq. (2) and Algorithm 1 ----
int dense_from_factors(const void *L, const void *R, void *M, int m, int dtype, cudaStream_t s);
int project_to_factors(const void *A, void *L, void *R, int m, int dtype, unsigned long long *rotations, cudaStream_t s);

// ---- elementwise steps of the feed-forward block's backward pass (mlp_bwd.cu) ----
// h = GELU(a (+ b1)); b1 may be null when a already holds the bias
int mlp_act(const void *a, const void *b1, void *h, float *zero1, float *zero2, int64_t tokens, int n, int dtype, cudaStream_t s);
// dh <- dh * GELU'(a (+ b1)) in place, db1 += column sums of the result, db2 += column sums of dy
int mlp_dact(void *dh, const void *a, const void *b1, const void *dy, float *db1, float *db2, int64_t tokens, int n,
             int dtype, cudaStream_t s);
// combination step of the complex multiply (planar tensors, plane_elems = tokens * n)
int cplx_combine(const void *A, const void *B, const void *C, const void *D, void *y, int64_t plane_elems, int adjoint,
                 int dtype, cudaStream_t s);
// fold the status word of an inner workspace into the outer one and clear it
int merge_status(unsigned *outer, unsigned *inner, cudaStream_t s);

}  // namespace monarch
