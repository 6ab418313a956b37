// Whole calls as one cooperative launch over "units" of block products (block_units.cu): the device code shared by the
// calls.  A call is a list of operations in phases; a phase's operations are cut into units that depend on nothing in
// the same phase, every CTA runs its share, and a grid barrier separates the phases.
//
// A unit of a stage is TT tokens x 8 neighbouring blocks x ES outputs of each block, one warp per block.  Eight blocks
// because the permutation P turns "block b, output e" into column e*m + b: eight blocks make 16 bytes (bf16) or 32
// bytes (fp32) of consecutive columns, so the permuted side is read and written in such pieces and re-ordered in
// shared memory.  The intermediates u, du between two stages are private to the library and are kept as
// mid[j/8][t][k][j%8], which both sides read and write in full lines.
//
// What bounds them: at a few tokens the chain of latencies of a phase (barrier, input from L2, product, result: 4 us
// per phase with the cold instruction fetches), which is why a phase's weights are fetched before its barrier; at many
// tokens the warps' issue of shared-memory accesses and legacy-shaped MMAs (ncu at 4096 tokens, m = 64: LSU data pipe
// 52 %, issue 29 %), which is why the kernels with weights in registers and the tcgen05 kernels take over there.  One CTA of 16 warps with a two-deep pipeline was
// no faster at any size than two CTAs of 8 warps whose loads overlap the other's work (23 against 27 us at 1000 tokens),
// and starting the permuted loads early cost spills (31 us).
#pragma once

#include <type_traits>

#include "common.cuh"

namespace monarch {
namespace units {

typedef __nv_bfloat16 bf16;

// What an operation does.  Roles of a tensor: kNat - block b is the major index of the row (columns b*m + c);
// kPerm - block b is the minor index (columns c*m + b).
enum Kind : int { kStage = 0, kWgrad = 1, kReduce = 2, kColsum = 3 };
enum Act : int { kNone = 0, kGelu = 1, kGeluGrad = 2 };

// How the pieces of 8 elements of a tensor are addressed, in pieces (32 bits: at most 2^20 tokens of 16384 elements):
// kNat: t * t_stride + b * b_stride + (c / 8) * c_stride;  kPerm: t * t_stride + (b / 8) * b_stride + c * c_stride.
struct View {
    void *p;
    unsigned t_stride, b_stride, c_stride;
    int mid;                 // the intermediate layout (decides which pieces are neighbours in memory)
};

struct Op {
    int kind, phase;
    int perm;                // role of the blocks in this operation's tensors
    int trans;               // stage: multiply by the transposed blocks
    int act, accumulate;
    int splits;              // wgrad: token ranges; > 1 leaves partial sums; reduce: number of parts
    View in, out;            // stage: input, output; wgrad: operand whose columns index the rows of the result; colsum: in
    View in2;                // wgrad: the other operand; stage: kGelu - where to leave the pre-activation (p may be
                             // null); kGeluGrad - the pre-activation
    const void *w;           // stage: weights [block][out][in]
    const void *bias;        // stage: bias by column or null
    float *sums;             // wgrad / reduce / colsum: result; stage with kGeluGrad: column sums per token tile
    const float *parts;      // reduce: parts, `count` apart
    long long count;         // reduce: elements
};

constexpr int kMaxOps = 18;
struct Params {
    Op op[kMaxOps];
    int n_ops, n_phases;
    int tokens;
    unsigned *status;        // [0] status word, [1] wait limit, [8] grid barrier, [9] CTAs done
};

constexpr int kBarrierWord = 8, kDoneWord = 9;
constexpr unsigned kErrGridWait = 0x301;

template <typename T_, int M_, int TT_, int ES_, int LS_, int KS_, int KC_ = 0> struct Cfg {
    typedef T_ T;
    static constexpr int M = M_, TT = TT_, ES = ES_, LS = LS_, KS = KS_, G = 8;
    static constexpr bool kBf = std::is_same<T, bf16>::value;
    static constexpr int kWpb = KC_ > 0 ? 2 : 1, kThreads = 32 * G * kWpb;   // warps per block
    static constexpr int EW = ES / kWpb, KW = KS / kWpb;      // outputs / gradient columns of one warp
    static constexpr int kPad = kBf ? 8 : 4;                  // rows 16 bytes longer: conflict-free ldmatrix / 16-byte reads
    static constexpr int PA = M + kPad, PE = kBf ? ES + kPad : ES, PL = LS + kPad, PK = KS + kPad;
    // KC > 0 (fp32, many tokens): both operands of a stage stream through shared memory, KC columns at a time, which
    // leaves room for 8 x 8 results per lane; one CTA per SM
    static constexpr int KC = KC_, PC = KC + 4;
    static constexpr int TW = KC ? 16 : 32;                   // tokens per step of a weight gradient
    static constexpr int cmax(int a, int b) { return a > b ? a : b; }
    // staging of results: permuted role - one plane of words per pair of bf16 blocks (per fp32 block), pitch 8 mod 32;
    // natural role - rows of ES outputs and rows of 8 blocks, each 16 bytes longer
    static constexpr int PS = ES + (40 - ES % 32) % 32, kPlanes = kBf ? G / 2 : G;
    static constexpr int kNatB = ES * (int)sizeof(T) + 16, kNatT = G * kNatB + 16;
    static constexpr int kStageBytes = cmax(kPlanes * TT * PS * 4, TT * kNatT);
    static constexpr int kTileBytes = G * TT * PA * (int)sizeof(T);
    static constexpr int kWBytes = cmax(G * ES * PA, G * M * PE) * (int)sizeof(T);
    static constexpr int kPadB = KC ? 4 : 0;                  // between the blocks of a step: 4-byte copies of 8 blocks without conflicts
    static constexpr int kBlockL = TW * PL + kPadB, kBlockK = TW * PK + kPadB;
    static constexpr int kStepBytes = G * (kBlockL + kBlockK) * (int)sizeof(T);
    // Two CTAs per SM work on different units while each waits for its own loads.  Within that share of shared memory: two
    // tiles (the next unit's input is on its way during this one's work), or one, or one that the results are staged over.
    static constexpr int kBlockA = TT * PC + 4, kChunkA = G * kBlockA * 4, kChunkW = cmax(G * ES * PC, G * KC * (ES + 4)) * 4, kChunk = kChunkA + kChunkW;
    static constexpr int kHalf = KC ? 226 * 1024 : 113 * 1024 - 512;
    static constexpr int kBufs = 2 * kTileBytes + kWBytes + kStageBytes <= kHalf ? 2 : 1;
    static constexpr bool kAlias = KC == 0 && kTileBytes + kWBytes + kStageBytes > kHalf;
    static constexpr int kWAt = kAlias ? cmax(kTileBytes, kStageBytes) : kBufs * kTileBytes;
    static constexpr int kStageAt = KC ? 2 * kChunk : kAlias ? 0 : kWAt + kWBytes;
    static constexpr int kStageSmem = kAlias ? kWAt + kWBytes : kStageAt + kStageBytes;
    static constexpr int kSteps = 2 * kStepBytes <= cmax(kStageSmem, kHalf) ? 2 : 1;   // buffers of a weight gradient
    static constexpr int kSmem = cmax(kStageSmem, kSteps * kStepBytes);
    static constexpr int kCtas = kSmem <= 113 * 1024 - 512 ? 2 : 1;
};

// ---------------------------------------------------------------- small device helpers
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2bf(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
template <typename T> struct Math;
template <> struct Math<bf16> {
    static __device__ __forceinline__ float gelu(float a) { return gelu_fast(a); }
    static __device__ __forceinline__ float grad(float a) { return gelu_fast_grad(a); }
};
template <> struct Math<float> {
    static __device__ __forceinline__ float gelu(float a) { return gelu_erf(a); }
    static __device__ __forceinline__ float grad(float a) { return gelu_erf_grad(a); }
};

// ---------------------------------------------------------------- loads into shared memory
// tile[b][t][c - 8 c8]: 8 blocks from b0 on, R tokens from t0 on (zeros past the last), NC columns from 8*c8 on.  begin()
// starts the transfer; end() finishes what goes through registers (the permuted role, which has to be re-ordered);
// afterwards cp_async_wait() and a barrier.
template <typename C, int R, int NC, int PITCH> struct TileLoad {
    typedef typename C::T T;
    static constexpr int kThreads = C::kThreads, H = (int)sizeof(T) / 2;         // 16-byte accesses per piece
    static constexpr int kTasks = R * NC / 2, U = (kTasks + kThreads - 1) / kThreads;
    uint4 lo[U][H], hi[U][H];

    // `left`: tokens from t0 on
    __device__ __forceinline__ void begin(T *tile, const View &v, int perm, int b0, int c8, int t0, int left)
    {
        const uint4 *src = static_cast<const uint4 *>(v.p);
        if (!perm) {
            // 16 bytes per lane, neighbours in memory on neighbouring lanes; per token: 8 blocks x NC / 8 pieces of H
            constexpr int kVecs = R * NC * H;
            const unsigned first = t0 * v.t_stride + b0 * v.b_stride + c8 * v.c_stride;
#pragma unroll 4
            for (int j = threadIdx.x; j < kVecs; j += kThreads) {
                const int h = j % H, i = j / H;
                int b, c;
                if (v.mid) { b = i % 8; c = i / 8 % (NC / 8); }
                else       { c = i % (NC / 8); b = i / (NC / 8) % 8; }
                const int t = i / NC;
                const bool ok = t < left;
                cp_async16(tile + (b * R + t) * PITCH + c * 8 + h * 4,
                           src + (size_t)(first + (ok ? t : 0) * v.t_stride + b * v.b_stride + c * v.c_stride) * H + h, ok);
            }
            return;
        }
        // pieces of 8 blocks: two columns per thread and task, so that bf16 is stored as pairs (a word of shared memory)
        const unsigned first = t0 * v.t_stride + b0 / 8 * v.b_stride + c8 * 8 * v.c_stride;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = u * kThreads + threadIdx.x, c = i % (NC / 2) * 2, t = i / (NC / 2);
            const bool ok = t < R && t < left;
            const unsigned g = first + (ok ? t : 0) * v.t_stride + c * v.c_stride;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                lo[u][h] = ok ? src[(size_t)g * H + h] : make_uint4(0, 0, 0, 0);
                hi[u][h] = ok ? src[(size_t)(g + v.c_stride) * H + h] : make_uint4(0, 0, 0, 0);
            }
        }
    }
    __device__ __forceinline__ void end(T *tile, int perm)
    {
        if (!perm) return;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = u * kThreads + threadIdx.x, c = i % (NC / 2) * 2, t = i / (NC / 2);
            if (t >= R) break;
            T *d = tile + t * PITCH + c;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t a[4] = {lo[u][h].x, lo[u][h].y, lo[u][h].z, lo[u][h].w};
                const uint32_t b[4] = {hi[u][h].x, hi[u][h].y, hi[u][h].z, hi[u][h].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if constexpr (H == 1) {
                        *reinterpret_cast<uint32_t *>(d + (2 * q) * R * PITCH) = __byte_perm(a[q], b[q], 0x5410);
                        *reinterpret_cast<uint32_t *>(d + (2 * q + 1) * R * PITCH) = __byte_perm(a[q], b[q], 0x7632);
                    } else {
                        *reinterpret_cast<uint2 *>(d + (4 * h + q) * R * PITCH) = make_uint2(a[q], b[q]);
                    }
                }
            }
        }
    }
};

// rows e0 .. e0 + ES of the result of 8 blocks in storage order, [b][e][c], of transposed blocks [b][c][e].  fp32: the ES / 8
// neighbouring rows of a lane are kept 8 rows apart, so that the lanes' reads fall on different banks.
template <typename C>
__device__ __forceinline__ void load_weights(typename C::T *wt, const void *w, int trans, int b0, int e0)
{
    typedef typename C::T T;
    constexpr int M = C::M, ES = C::ES, V = 16 / (int)sizeof(T);
    const T *src = static_cast<const T *>(w) + (size_t)b0 * M * M;
    if (!trans) {
        constexpr int kVecs = 8 * ES * (M / V);
#pragma unroll 4
        for (int i = threadIdx.x; i < kVecs; i += C::kThreads) {
            const int c = i % (M / V) * V, e = i / (M / V) % ES, b = i / (M / V * ES);
            const int row = C::kBf ? e : e % (ES / 8) * 8 + e / (ES / 8);
            cp_async16(wt + (b * ES + row) * C::PA + c, src + ((size_t)b * M + e0 + e) * M + c, true);
        }
    } else {
        constexpr int kVecs = 8 * M * (ES / V);
#pragma unroll 4
        for (int i = threadIdx.x; i < kVecs; i += C::kThreads) {
            const int e = i % (ES / V) * V, c = i / (ES / V) % M, b = i / (ES / V * M);
            cp_async16(wt + (b * M + c) * C::PE + e, src + ((size_t)b * M + c) * M + e0 + e, true);
        }
    }
}

// ---------------------------------------------------------------- results of a stage unit
// Accumulators of one warp (TT tokens, EW outputs of its block), visited with their token and output numbers.
template <typename C, bool BF = C::kBf> struct Acc;
template <typename C> struct Acc<C, true> {
    float v[C::TT / 16][C::EW / 8][4];
    template <typename F> __device__ __forceinline__ void each(F f)
    {
        const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
#pragma unroll
        for (int mt = 0; mt < C::TT / 16; ++mt)
#pragma unroll
            for (int nt = 0; nt < C::EW / 8; ++nt)
#pragma unroll
                for (int r = 0; r < 4; ++r) f(v[mt][nt][r], mt * 16 + g + (r >> 1) * 8, nt * 8 + 2 * q + (r & 1));
    }
    // f(sum over the tile's tokens, output) in one lane per output
    template <typename F> __device__ __forceinline__ void column_sums(F f)
    {
        const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
#pragma unroll
        for (int nt = 0; nt < C::EW / 8; ++nt)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                float s = 0.0f;
#pragma unroll
                for (int mt = 0; mt < C::TT / 16; ++mt) s += v[mt][nt][p] + v[mt][nt][p + 2];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (g == 0) f(s, nt * 8 + 2 * q + p);
            }
    }
};
template <typename C> struct Acc<C, false> {
    float v[C::TT / 4][C::EW / 8];
    static constexpr int V = C::EW / 8 < 4 ? C::EW / 8 : 4;
    int packed;                                        // KC > 0: outputs of a lane are V neighbours at a time, else every eighth
    __device__ __forceinline__ int output(int el, int q) const { return C::KC == 0 || packed ? V * el + 8 * V * (q / V) + q % V : el + 8 * q; }
    template <typename F> __device__ __forceinline__ void each(F f)
    {
        const int tl = (threadIdx.x & 31) >> 3, el = threadIdx.x & 7;
#pragma unroll
        for (int i = 0; i < C::TT / 4; ++i)
#pragma unroll
            for (int q = 0; q < C::EW / 8; ++q) f(v[i][q], tl + 4 * i, output(el, q));
    }
    template <typename F> __device__ __forceinline__ void column_sums(F f)
    {
        const int tl = (threadIdx.x & 31) >> 3, el = threadIdx.x & 7;
#pragma unroll
        for (int q = 0; q < C::EW / 8; ++q) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < C::TT / 4; ++i) s += v[i][q];
            s += __shfl_xor_sync(0xffffffffu, s, 8);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (tl == 0) f(s, output(el, q));
        }
    }
};

__device__ __forceinline__ uint32_t f2w(float x) { return __float_as_uint(x); }

// Accumulators -> storage type -> staging in shared memory (stage_results), then, after a barrier, staging -> global
// memory in pieces of 8 elements (copy_out).  The permuted role needs the 8 blocks of one (token, output) side by side,
// one value from each warp: hence the planes, whose pitch keeps both sides free of bank conflicts.
template <typename C> __device__ __forceinline__ void stage_results(Acc<C> &acc, unsigned char *stage, int perm)
{
    const int w = threadIdx.x >> 5, b = w / C::kWpb, e0 = w % C::kWpb * C::EW;
    if constexpr (!C::kBf && C::KC == 0) {             // a lane's outputs are neighbours
        constexpr int V = C::ES / 8;
        static_assert(V == 2 || V == 4, "");
        const int tl = (threadIdx.x & 31) >> 3, el = threadIdx.x & 7;
#pragma unroll
        for (int i = 0; i < C::TT / 4; ++i) {
            const int t = tl + 4 * i;
            unsigned char *to = perm ? stage + ((b * C::TT + t) * C::PS + V * el) * 4 : stage + t * C::kNatT + b * C::kNatB + V * el * 4;
            if constexpr (V == 4) *reinterpret_cast<float4 *>(to) = make_float4(acc.v[i][0], acc.v[i][1], acc.v[i][2], acc.v[i][3]);
            else                  *reinterpret_cast<float2 *>(to) = make_float2(acc.v[i][0], acc.v[i][1]);
        }
        return;
    }
    if (!perm) {
        if constexpr (C::kBf) {
            const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
#pragma unroll
            for (int mt = 0; mt < C::TT / 16; ++mt)
#pragma unroll
                for (int nt = 0; nt < C::EW / 8; ++nt)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<uint32_t *>(stage + (mt * 16 + g + 8 * h) * C::kNatT + b * C::kNatB + (e0 + nt * 8 + 2 * q) * 2) =
                            pack2bf(acc.v[mt][nt][2 * h], acc.v[mt][nt][2 * h + 1]);
        } else {
            acc.each([&](float v, int t, int e) { *reinterpret_cast<float *>(stage + t * C::kNatT + b * C::kNatB + (e0 + e) * 4) = v; });
        }
    } else if constexpr (C::kBf) {
        acc.each([&](float v, int t, int e) {
            reinterpret_cast<bf16 *>(stage)[(((b >> 1) * C::TT + t) * C::PS + e0 + e) * 2 + (b & 1)] = __float2bfloat16_rn(v);
        });
    } else {
        acc.each([&](float v, int t, int e) { reinterpret_cast<float *>(stage)[(b * C::TT + t) * C::PS + e0 + e] = v; });
    }
}

template <typename C>
__device__ __forceinline__ void copy_out(const unsigned char *stage, const View &out, int perm, int b0, int e0, int t0, int left)
{
    typedef typename C::T T;
    constexpr int H = (int)sizeof(T) / 2;
    uint4 *dst = static_cast<uint4 *>(out.p);
    constexpr int kVecs = C::TT * C::ES * H;           // natural: per token 8 blocks x ES / 8 pieces; permuted: ES; H each
    if (!perm) {
        const unsigned first = t0 * out.t_stride + b0 * out.b_stride + e0 / 8 * out.c_stride;
#pragma unroll 4
        for (int j = threadIdx.x; j < kVecs; j += C::kThreads) {
            const int h = j % H, i = j / H;
            int b, c;
            if (out.mid) { b = i % 8; c = i / 8 % (C::ES / 8); }
            else         { c = i % (C::ES / 8); b = i / (C::ES / 8) % 8; }
            const int t = i / C::ES;
            if (t >= left) break;
            dst[(size_t)(first + t * out.t_stride + b * out.b_stride + c * out.c_stride) * H + h] =
                *reinterpret_cast<const uint4 *>(stage + t * C::kNatT + b * C::kNatB + c * 8 * sizeof(T) + h * 16);
        }
        return;
    }
    const unsigned first = t0 * out.t_stride + b0 / 8 * out.b_stride + e0 * out.c_stride;
#pragma unroll 4
    for (int j = threadIdx.x; j < kVecs; j += C::kThreads) {
        const int h = j % H, e = j / H % C::ES, t = j / (H * C::ES);
        if (t >= left) break;
        constexpr int kPlane = C::TT * C::PS;
        const uint32_t *s = reinterpret_cast<const uint32_t *>(stage) + h * 4 * kPlane + t * C::PS + e;
        dst[(size_t)(first + t * out.t_stride + e * out.c_stride) * H + h] = make_uint4(s[0], s[kPlane], s[2 * kPlane], s[3 * kPlane]);
    }
}

// ---------------------------------------------------------------- a stage unit
// fp32, transposed blocks, whose columns are rows of shared memory: fma.rn.f32x2 takes two neighbouring outputs; partial sums over
// even and odd columns as below.  (Transposed on their way into shared memory, through registers, dx of 200 tokens at m = 64
// took 36 us, of 24 tokens at m = 128 37; now 31 and 29.)
template <typename C> __device__ __forceinline__ Acc<C> multiply_transposed(const float *tile, const float *wt)
{
    constexpr int M = C::M, TT = C::TT, RE = C::EW / 8;
    const int b = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Acc<C> acc;
    const float *a = tile + (b * TT + (lane >> 3)) * C::PA, *bw = wt + b * M * C::PE + RE * (lane & 7);
    f32x2 s[2][TT / 4][RE / 2];
#pragma unroll
    for (int i = 0; i < TT / 4; ++i)
#pragma unroll
        for (int q = 0; q < RE / 2; ++q) s[0][i][q] = s[1][i][q] = 0;
#pragma unroll 1
    for (int c = 0; c < M; c += 4) {
        f32x2 fb[4][RE / 2];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (RE == 4) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(bw + (c + k) * C::PE);
                fb[k][0] = t.x;
                fb[k][1] = t.y;
            } else {
                fb[k][0] = *reinterpret_cast<const f32x2 *>(bw + (c + k) * C::PE);
            }
        }
#pragma unroll
        for (int i = 0; i < TT / 4; ++i) {
            const float4 fa = *reinterpret_cast<const float4 *>(a + 4 * i * C::PA + c);
            const float av[4] = {fa.x, fa.y, fa.z, fa.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int q = 0; q < RE / 2; ++q) s[k & 1][i][q] = fma2(pack2(av[k], av[k]), fb[k][q], s[k & 1][i][q]);
        }
    }
#pragma unroll
    for (int i = 0; i < TT / 4; ++i)
#pragma unroll
        for (int q = 0; q < RE / 2; ++q) {
            const float2 even = unpack2(s[0][i][q]), odd = unpack2(s[1][i][q]);
            acc.v[i][2 * q] = even.x + odd.x;
            acc.v[i][2 * q + 1] = even.y + odd.y;
        }
    return acc;
}
// out of line: inlined beside the other product it costs m = 128 registers (dx of 24 tokens 31 us, forward 26.6; so 28.8 and 24.7)
template <typename C> __device__ __noinline__ Acc<C> multiply_transposed_far(const float *tile, const float *wt) { return multiply_transposed<C>(tile, wt); }

template <typename C>
__device__ __forceinline__ void multiply(Acc<C> &acc, const typename C::T *tile, const typename C::T *wt, int trans)
{
    constexpr int M = C::M, TT = C::TT, ES = C::ES, EW = C::EW;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, b = w / C::kWpb, e0 = w % C::kWpb * EW;
    if constexpr (C::kBf) {
#pragma unroll
        for (int mt = 0; mt < TT / 16; ++mt)
#pragma unroll
            for (int nt = 0; nt < EW / 8; ++nt)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc.v[mt][nt][r] = 0.0f;
        const bf16 *a = tile + (b * TT + (lane & 15)) * C::PA + (lane >> 4) * 8;
        // with 8 outputs per warp one ldmatrix brings two steps of the contraction, otherwise two groups of 8 outputs
        constexpr bool kPair = EW >= 16;
        const bf16 *bn = wt + (b * ES + e0 + (lane & 7) + (kPair ? (lane >> 4) * 8 : 0)) * C::PA + (kPair ? lane >> 3 & 1 : lane >> 3) * 8;
        const bf16 *bt = wt + (b * M + (kPair ? lane & 15 : lane)) * C::PE + e0 + (kPair ? (lane >> 4) * 8 : 0);
        uint32_t keep[2];
#pragma unroll
        for (int ks = 0; ks < M / 16; ++ks) {
            uint32_t fa[TT / 16][4];
#pragma unroll
            for (int mt = 0; mt < TT / 16; ++mt) ldsm4(fa[mt], a + mt * 16 * C::PA + ks * 16);
            if constexpr (kPair) {
#pragma unroll
                for (int np = 0; np < EW / 16; ++np) {
                    uint32_t fb[4];
                    if (trans) ldsm4_trans(fb, bt + ks * 16 * C::PE + np * 16);
                    else       ldsm4(fb, bn + np * 16 * C::PA + ks * 16);
#pragma unroll
                    for (int mt = 0; mt < TT / 16; ++mt) {
                        mma16816(acc.v[mt][2 * np], fa[mt], fb[0], fb[1]);
                        mma16816(acc.v[mt][2 * np + 1], fa[mt], fb[2], fb[3]);
                    }
                }
            } else if constexpr (M == 16) {            // a single step: both halves of the lanes fetch the same 16 columns
                uint32_t fb[4];
                if (trans) ldsm4_trans(fb, wt + (b * M + (lane & 15)) * C::PE + e0);
                else       ldsm4(fb, wt + (b * ES + e0 + (lane & 7)) * C::PA + (lane >> 3 & 1) * 8);
#pragma unroll
                for (int mt = 0; mt < TT / 16; ++mt) mma16816(acc.v[mt][0], fa[mt], fb[0], fb[1]);
            } else {
                uint32_t b0 = keep[0], b1 = keep[1];
                if (ks % 2 == 0) {
                    uint32_t fb[4];
                    if (trans) ldsm4_trans(fb, bt + ks * 16 * C::PE);
                    else       ldsm4(fb, bn + ks * 16);
                    b0 = fb[0];
                    b1 = fb[1];
                    keep[0] = fb[2];
                    keep[1] = fb[3];
                }
#pragma unroll
                for (int mt = 0; mt < TT / 16; ++mt) mma16816(acc.v[mt][0], fa[mt], b0, b1);
            }
        }
    } else {
        // two partial sums per result (even and odd columns), packed for fma.rn.f32x2
        if (trans) {
            const Acc<C> t = M == 128 ? multiply_transposed_far<C>(tile, wt) : multiply_transposed<C>(tile, wt);
#pragma unroll
            for (int i = 0; i < TT / 4; ++i)
#pragma unroll
                for (int q = 0; q < EW / 8; ++q) acc.v[i][q] = t.v[i][q];
            return;
        }
        const float *a = tile + (b * TT + (lane >> 3)) * C::PA, *bw = wt + (b * ES + (lane & 7)) * C::PA;
        f32x2 s[TT / 4][EW / 8];
#pragma unroll
        for (int i = 0; i < TT / 4; ++i)
#pragma unroll
            for (int q = 0; q < EW / 8; ++q) s[i][q] = 0;
#pragma unroll 2
        for (int c = 0; c < M; c += 4) {
            ulonglong2 fb[EW / 8];
#pragma unroll
            for (int q = 0; q < EW / 8; ++q) fb[q] = *reinterpret_cast<const ulonglong2 *>(bw + 8 * q * C::PA + c);
#pragma unroll
            for (int i = 0; i < TT / 4; ++i) {
                const ulonglong2 fa = *reinterpret_cast<const ulonglong2 *>(a + 4 * i * C::PA + c);
#pragma unroll
                for (int q = 0; q < EW / 8; ++q) s[i][q] = fma2(fa.y, fb[q].y, fma2(fa.x, fb[q].x, s[i][q]));
            }
        }
#pragma unroll
        for (int i = 0; i < TT / 4; ++i)
#pragma unroll
            for (int q = 0; q < EW / 8; ++q) {
                const float2 t = unpack2(s[i][q]);
                acc.v[i][q] = t.x + t.y;
            }
    }
}

// NC columns from c0 on of R tokens and 8 blocks to tile[block][token][column] (fp32, asynchronous; rows PITCH, blocks BLOCK
// floats apart): permuted pieces (8 blocks, 32 bytes) go to the blocks' rows 4 bytes at a time.  A thread's pieces differ in
// the token only: one address and an add per piece.
template <typename C, int R, int NC, int PITCH, int BLOCK>
__device__ __forceinline__ void load_async(float *tile, const View &v, int perm, int b0, int c0, int t0, int left)
{
    const unsigned j = threadIdx.x;
    if (!perm) {
        constexpr int kStep = C::kThreads / (2 * NC);
        const unsigned h = j % 2, i = j / 2, t = i / NC;
        const unsigned b = v.mid ? i % 8 : i / (NC / 8) % 8, c = v.mid ? i / 8 % (NC / 8) : i % (NC / 8);
        const float4 *src = static_cast<const float4 *>(v.p) +
                            (size_t)((t0 + t) * v.t_stride + (b0 + b) * v.b_stride + (c0 / 8 + c) * v.c_stride) * 2 + h;
        float *dst = tile + b * BLOCK + t * PITCH + c * 8 + h * 4;
        if (left >= R) {                                   // (most tiles are whole)
#pragma unroll
            for (int n = 0; n < R / kStep; ++n, src += (size_t)kStep * v.t_stride * 2) cp_async16(dst + n * kStep * PITCH, src, true);
            return;
        }
#pragma unroll 1
        for (int n = 0; n < R / kStep; ++n) {
            const bool ok = (int)t + n * kStep < left;
            cp_async16(dst + n * kStep * PITCH, ok ? src + (size_t)n * kStep * v.t_stride * 2 : static_cast<const float4 *>(v.p), ok);
        }
        return;
    }
    constexpr int kStep = C::kThreads / (8 * NC);
    static_assert(kStep >= 1 && R % kStep == 0, "");
    const unsigned b = j % 8, c = j / 8 % NC, t = j / (8 * NC);
    const float *src = static_cast<const float *>(v.p) + (size_t)((t0 + t) * v.t_stride + b0 / 8 * v.b_stride + (c0 + c) * v.c_stride) * 8 + b;
    const uint32_t dst = smem_addr(tile + b * BLOCK + t * PITCH + c);
    if (left >= R) {
#pragma unroll
        for (int n = 0; n < R / kStep; ++n, src += (size_t)kStep * v.t_stride * 8)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + n * kStep * PITCH * 4), "l"(src) : "memory");
        return;
    }
#pragma unroll 1
    for (int n = 0; n < R / kStep; ++n) {
        const bool ok = (int)t + n * kStep < left;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + n * kStep * PITCH * 4),
                     "l"(ok ? src + (size_t)n * kStep * v.t_stride * 8 : static_cast<const float *>(v.p)), "r"(ok ? 4 : 0) : "memory");
    }
}

// ---- the same with both operands streamed in chunks of KC columns (fp32, many tokens)
// Bound by FMA issue once a lane has 8 x 4 results: 12 loads of 16 bytes from shared memory feed 64 packed FMAs, where the
// 4 x 4 results that fit beside resident operands take 8 for 32 and wait for shared memory (m = 64, us: forward of 1500
// tokens 158 -> 107, forward + backward of 2048 tokens 544 -> 397; m = 128, 400 tokens 997 -> 742; m = 32, 8000 tokens
// 379 -> 331).  Blocks as stored ([out][in]): the FMA packs two columns of the contraction; transposed blocks ([in][out]):
// it packs two outputs.
template <typename C> struct Chunks {
    static constexpr int TT = C::TT, ES = C::ES, KC = C::KC, PC = C::PC, M = C::M, EW = C::EW, RT = TT / 4, RE = EW / 8;
    static_assert(KC % 8 == 0, "a half of a chunk is multiplied four columns at a time");
    f32x2 s[RT][RE];                                   // [out][in]: sums over even and odd columns; else [RT][RE / 2] used

    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int q = 0; q < RE; ++q) s[i][q] = 0;
    }
    static __device__ __forceinline__ void load_w(float *wt, const void *w, int trans, int b0, int e0, int c0)
    {
        const float *src = static_cast<const float *>(w) + (size_t)b0 * M * M;
        const unsigned j = threadIdx.x;
        constexpr int kPer = ES * KC / 4, kStep = C::kThreads / kPer;      // pieces of a block, blocks per step
        const unsigned c = trans ? j / (ES / 4) % KC : j % (KC / 4) * 4, e = trans ? j % (ES / 4) * 4 : j / (KC / 4) % ES, b = j / kPer;
        src += (b * M + (trans ? c0 + c : e0 + e)) * M + (trans ? e0 + e : c0 + c);
        float *dst = wt + (trans ? (b * KC + c) * (ES + 4) + e : (b * ES + e) * PC + c);
        const int step = trans ? kStep * KC * (ES + 4) : kStep * ES * PC;
        static_assert(C::kThreads % kPer == 0 && 8 % kStep == 0, "");
#pragma unroll
        for (int n = 0; n < 8 / kStep; ++n) cp_async16(dst + n * step, src + (size_t)n * kStep * M * M, true);
    }
    // the columns of one half of a chunk
    __device__ __forceinline__ void multiply(const float *tile, const float *wt, int trans, int half)
    {
        const int w = (threadIdx.x >> 5) / C::kWpb, e0 = (threadIdx.x >> 5) % C::kWpb * EW;
        const int tl = (threadIdx.x & 31) >> 3, el = threadIdx.x & 7;
        const float *a = tile + w * C::kBlockA + tl * PC + half * (KC / 2);
        if (!trans) {
            const float *b = wt + (w * ES + e0 + el) * PC + half * (KC / 2);
#pragma unroll
            for (int c = 0; c < KC / 2; c += 4) {
                ulonglong2 fb[RE];
#pragma unroll
                for (int q = 0; q < RE; ++q) fb[q] = *reinterpret_cast<const ulonglong2 *>(b + 8 * q * PC + c);
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const ulonglong2 fa = *reinterpret_cast<const ulonglong2 *>(a + 4 * i * PC + c);
#pragma unroll
                    for (int q = 0; q < RE; ++q) s[i][q] = fma2(fa.y, fb[q].y, fma2(fa.x, fb[q].x, s[i][q]));
                }
            }
        } else {
            constexpr int V = RE < 4 ? RE : 4;             // neighbouring outputs of a lane
            const float *b = wt + (w * KC + half * (KC / 2)) * (ES + 4) + e0 + V * el;
#pragma unroll
            for (int c = 0; c < KC / 2; c += 4) {
                f32x2 fb[4][RE / 2];
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int q = 0; q < RE / V; ++q) {
                        const float *at = b + (c + k) * (ES + 4) + 8 * V * q;
                        if constexpr (V == 4) {
                            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(at);
                            fb[k][2 * q] = t.x;
                            fb[k][2 * q + 1] = t.y;
                        } else {
                            fb[k][q] = *reinterpret_cast<const f32x2 *>(at);
                        }
                    }
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const float4 fa = *reinterpret_cast<const float4 *>(a + 4 * i * PC + c);
                    const float av[4] = {fa.x, fa.y, fa.z, fa.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const f32x2 d = pack2(av[k], av[k]);
#pragma unroll
                        for (int q = 0; q < RE / 2; ++q) s[i][q] = fma2(d, fb[k][q], s[i][q]);
                    }
                }
            }
        }
    }
    __device__ __forceinline__ void finish(Acc<C> &acc, int trans) const
    {
        acc.packed = trans;
        if (trans) {
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int q = 0; q < RE / 2; ++q) {
                    const float2 t = unpack2(s[i][q]);
                    acc.v[i][2 * q] = t.x;
                    acc.v[i][2 * q + 1] = t.y;
                }
        } else {
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int q = 0; q < RE; ++q) {
                    const float2 t = unpack2(s[i][q]);
                    acc.v[i][q] = t.x + t.y;
                }
        }
    }
};

// bias, activation, staging and the copy to memory: shared by both forms.  On return the results are staged and a
// barrier has been passed; the caller copies them out (copy_out) when it has started its next loads.
template <typename C>
__device__ __forceinline__ void finish_unit(const Op &op, Acc<C> &acc, unsigned char *stage, int b0, int e0, int tile_no, int tokens)
{
    typedef typename C::T T;
    constexpr int M = C::M, N = M * M;
    const int w = threadIdx.x >> 5, t0 = tile_no * C::TT, left = tokens - t0;
    const int b = b0 + w / C::kWpb, ew = e0 + w % C::kWpb * C::EW;
    if (op.bias != nullptr) {
        const T *bias = static_cast<const T *>(op.bias);
        acc.each([&](float &v, int, int e) { v += elem<T>::load(bias + (op.perm ? (ew + e) * M + b : b * M + ew + e)); });
    }
    if (C::kAlias) __syncthreads();                    // every warp is done with the tile
    if (op.act == kGelu) {
        if (op.in2.p != nullptr) {
            stage_results<C>(acc, stage, op.perm);
            __syncthreads();
            copy_out<C>(stage, op.in2, op.perm, b0, e0, t0, left);
            __syncthreads();
        }
        acc.each([&](float &v, int, int) { v = Math<T>::gelu(v); });
    } else if (op.act == kGeluGrad) {
        const T *a = static_cast<const T *>(op.in2.p);
        acc.each([&](float &v, int t, int e) {
            v = t < left ? v * Math<T>::grad(elem<T>::load(a + (size_t)(t0 + t) * N + b * M + ew + e)) : 0.0f;   // (0 x Inf of padding)
        });
        acc.column_sums([&](float s, int e) { op.sums[(size_t)tile_no * N + b * M + ew + e] = s; });
    }
    stage_results<C>(acc, stage, op.perm);
    __syncthreads();                                   // results staged; nobody reads the tile or the weights any more
}

// Units i0 .. i1 of a stage, in order: (8 blocks, ES outputs) major, token tile minor.  `held`: whose weights are in
// shared memory.
template <typename C>
__device__ __forceinline__ void stage_units(const Op &op, int i0, int i1, int tiles, int tokens, unsigned char *smem, int &held)
{
    typedef typename C::T T;
    constexpr int M = C::M, kSlices = M / C::ES;
    T *wt = reinterpret_cast<T *>(smem + C::kWAt);
    unsigned char *stage = smem + C::kStageAt;
    TileLoad<C, C::TT, M, C::PA> load;
    int at = i0 / tiles, tile_no = i0 % tiles, buf = 0;
    __syncthreads();                                   // what ran before has left shared memory
    if (held != at) {
        load_weights<C>(wt, op.w, op.trans, at / kSlices * 8, at % kSlices * C::ES);
        held = at;
    }
    load.begin(reinterpret_cast<T *>(smem), op.in, op.perm, at / kSlices * 8, 0, tile_no * C::TT, tokens - tile_no * C::TT);
    load.end(reinterpret_cast<T *>(smem), op.perm);
    for (int i = i0; i < i1; ++i) {
        const int b0 = at / kSlices * 8, e0 = at % kSlices * C::ES;
        const int t0 = tile_no * C::TT, left = tokens - t0, this_tile = tile_no;
        T *tile = reinterpret_cast<T *>(smem + buf * C::kTileBytes);
        const bool more = i + 1 < i1;
        if (++tile_no == tiles) { tile_no = 0; ++at; }
        if (C::kBufs == 2) buf ^= 1;
        T *next = reinterpret_cast<T *>(smem + buf * C::kTileBytes);
        cp_async_wait();
        __syncthreads();                               // tile and weights are here; the last results have been copied out
        // (what goes through registers starts late: held across the product it would cost more than it hides)
        const bool early = more && C::kBufs == 2 && !op.perm;
        if (early) load.begin(next, op.in, op.perm, at / kSlices * 8, 0, tile_no * C::TT, tokens - tile_no * C::TT);
        Acc<C> acc;
        multiply<C>(acc, tile, wt, op.trans);
        finish_unit<C>(op, acc, stage, b0, e0, this_tile, tokens);
        if (more) {
            if (held != at) {
                load_weights<C>(wt, op.w, op.trans, at / kSlices * 8, at % kSlices * C::ES);
                held = at;
            }
            if (!early && !C::kAlias) load.begin(next, op.in, op.perm, at / kSlices * 8, 0, tile_no * C::TT, tokens - tile_no * C::TT);
        }
        copy_out<C>(stage, op.out, op.perm, b0, e0, t0, left);
        if (C::kAlias && more) {
            __syncthreads();                           // the staged results have been read
            if (!early) load.begin(next, op.in, op.perm, at / kSlices * 8, 0, tile_no * C::TT, tokens - tile_no * C::TT);
        }
        if (more) load.end(next, op.perm);
    }
}

// part of PARTS of copy_out
template <typename C, int PARTS>
__device__ __forceinline__ void copy_part(const unsigned char *stage, const View &out, int perm, int b0, int e0, int t0, int left, int part)
{
    constexpr int ES = C::ES, kTok = C::TT / PARTS, kStep = C::kThreads / (2 * ES), kPlane = C::TT * C::PS;
    static_assert(C::kThreads % (2 * ES) == 0 && kTok % kStep == 0, "");
    const unsigned j = threadIdx.x, h = j % 2, i = j / 2 % ES, t = part * kTok + j / (2 * ES);
    const unsigned b = perm ? 0 : out.mid ? i % 8 : i / (ES / 8), c = perm ? i : out.mid ? i / 8 : i % (ES / 8);
    uint4 *dst = static_cast<uint4 *>(out.p) +
                 (size_t)((t0 + t) * out.t_stride + (perm ? b0 / 8 : b0 + b) * out.b_stride + ((perm ? e0 : e0 / 8) + c) * out.c_stride) * 2 + h;
    const unsigned char *from = stage + (perm ? (h * 4 * kPlane + t * C::PS + c) * 4 : t * C::kNatT + b * C::kNatB + c * 32 + h * 16);
#pragma unroll
    for (int n = 0; n < kTok / kStep; ++n, dst += (size_t)kStep * out.t_stride * 2) {
        if ((int)t + n * kStep >= left) break;
        if (perm) {
            const uint32_t *s = reinterpret_cast<const uint32_t *>(from) + n * kStep * C::PS;
            *dst = make_uint4(s[0], s[kPlane], s[2 * kPlane], s[3 * kPlane]);
        } else {
            *dst = *reinterpret_cast<const uint4 *>(from + n * kStep * C::kNatT);
        }
    }
}

template <typename C>
__device__ __forceinline__ void stage_units_chunked(const Op &op, int i0, int i1, int tiles, int tokens, unsigned char *smem)
{
    constexpr int M = C::M, kSlices = M / C::ES, KC = C::KC, kChunks = M / KC;
    unsigned char *stage = smem + C::kStageAt;
    struct Unit {
        int at, tile_no;
        __device__ __forceinline__ int b0() const { return at / kSlices * 8; }
        __device__ __forceinline__ int e0() const { return at % kSlices * C::ES; }
        __device__ __forceinline__ int t0() const { return tile_no * C::TT; }
    };
    auto after = [&](Unit u) { return u.tile_no + 1 == tiles ? Unit{u.at + 1, 0} : Unit{u.at, u.tile_no + 1}; };
    auto tile = [&](int n) { return reinterpret_cast<float *>(smem + (n & 1) * C::kChunk); };
    auto wt = [&](int n) { return reinterpret_cast<float *>(smem + (n & 1) * C::kChunk + C::kChunkA); };
    auto begin = [&](int n, Unit u, int k) {
        load_async<C, C::TT, KC, C::PC, C::kBlockA>(tile(n), op.in, op.perm, u.b0(), k * KC, u.t0(), tokens - u.t0());
        Chunks<C>::load_w(wt(n), op.w, op.trans, u.b0(), u.e0(), k * KC);
    };
    constexpr int kParts = kChunks / 2;
    auto copy = [&](Unit u, int part) {
        copy_part<C, kParts>(stage, op.out, op.perm, u.b0(), u.e0(), u.t0(), tokens - u.t0(), part);
    };
    // Of the four warps of a scheduler two start the next loads before their products and two between the halves of theirs: with
    // all of them in step the FMAs of a chunk and the address arithmetic of the next one followed one another (forward of 2048
    // tokens at m = 64 113 -> 106 us, forward + backward at m = 32, 8000 tokens, 226 -> 208; a quarter each: 107 and 209, and at
    // m = 128, 500 tokens, forward + backward 741 where halves take 711).
    const int mine = threadIdx.x >> 7 & 1;
    int n = 0;
    Unit u = {i0 / tiles, i0 % tiles}, last = u;
    __syncthreads();                                   // what ran before has left shared memory
    begin(0, u, 0);
    for (int i = i0; i < i1; ++i) {
        Chunks<C> sums;
        sums.clear();
        const Unit next = after(u);
#pragma unroll 1
        for (int k = 0; k < kChunks; ++k, ++n) {
            cp_async_wait();
            __syncthreads();                           // chunk n is here, chunk n - 1 has been read
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                if (half == mine) {
                    if (k + 1 < kChunks)  begin(n + 1, u, k + 1);
                    else if (i + 1 < i1)  begin(n + 1, next, 0);
                    // the previous unit's results leave during the first half of this one's products
                    if (i > i0 && k < kParts) copy(last, k);
                }
                sums.multiply(tile(n), wt(n), op.trans, half);
            }
        }
        Acc<C> acc;
        sums.finish(acc, op.trans);
        finish_unit<C>(op, acc, stage, u.b0(), u.e0(), u.tile_no, tokens);
        last = u;
        u = next;
    }
    for (int part = 0; part < kParts; ++part) copy(last, part);
}

// ---------------------------------------------------------------- a weight-gradient unit
// sums[b][l][k] = sum over a range of tokens of in[t](b, l) in2[t](b, k), for 8 blocks, LS rows and KS columns
template <typename C>
__device__ __forceinline__ void wgrad_unit(const Op &op, int b0, int l0, int k0, int split, int tokens, unsigned char *smem)
{
    typedef typename C::T T;
    constexpr int M = C::M, LS = C::LS, KS = C::KS, KW = C::KW, TW = C::TW;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, bw = w / C::kWpb, kw = w % C::kWpb * KW;
    const int steps = (tokens + TW - 1) / TW, per = (steps + op.splits - 1) / op.splits;
    const int s0 = split * per, s1 = s0 + per < steps ? s0 + per : steps;
    float *dst = op.sums + (op.splits > 1 ? (size_t)split * M * M * M : 0) + (size_t)(b0 + bw) * M * M + (size_t)l0 * M + k0 + kw;
    const bool add = op.splits == 1 && op.accumulate;
    constexpr int kMask = C::kSteps - 1;
    static_assert(C::KC == 0 || (C::kSteps == 2 && !C::kBf && C::TW > 1), "half of the warps load in the middle of a step, into the other buffer");
    TileLoad<C, TW, LS, C::PL> load_a;
    TileLoad<C, TW, KS, C::PK> load_b;
    auto tile_a = [&](int buf) { return reinterpret_cast<T *>(smem + buf * C::kStepBytes); };
    auto tile_b = [&](int buf) { return tile_a(buf) + C::G * C::kBlockL; };
    // operands of the natural role are asynchronous; the others go through registers, one operand after the other, unless many
    // fp32 tokens make the copies of 4 bytes worth their number
    auto load = [&](int s) {
        if constexpr (C::KC > 0) {
            load_async<C, TW, LS, C::PL, C::kBlockL>(tile_a(s & kMask), op.in, op.perm, b0, l0, s * TW, tokens - s * TW);
            load_async<C, TW, KS, C::PK, C::kBlockK>(tile_b(s & kMask), op.in2, op.perm, b0, k0, s * TW, tokens - s * TW);
            return;
        }
        load_a.begin(tile_a(s & kMask), op.in, op.perm, b0, l0 / 8, s * TW, tokens - s * TW);
        load_a.end(tile_a(s & kMask), op.perm);
        load_b.begin(tile_b(s & kMask), op.in2, op.perm, b0, k0 / 8, s * TW, tokens - s * TW);
        load_b.end(tile_b(s & kMask), op.perm);
    };
    constexpr int RL = LS / 4, RK = KW / 8;            // fp32: rows and columns of a lane, the columns VK neighbours at a time
    constexpr int VK = RK < 4 ? RK : 4;
    float acc[C::kBf ? LS / 16 : RL][C::kBf ? KW / 8 : RK][C::kBf ? 4 : 1] = {};

    __syncthreads();                                   // what ran before has left shared memory
    if (s0 < s1) load(s0);
#pragma unroll 1
    for (int s = s0; s < s1; ++s) {
        cp_async_wait();
        __syncthreads();                               // the operands of s are here, those of s - 1 have been read
        const bool early = C::kSteps == 2 && (C::KC > 0 || !op.perm);
        const int mine = C::KC > 0 ? threadIdx.x >> 7 & 1 : 0;    // (as in stage_units_chunked)
        if (early && s + 1 < s1 && mine == 0) load(s + 1);
        if constexpr (C::kBf) {
            const bf16 *a = tile_a(s & kMask) + (bw * TW + (lane & 7) + (lane >> 4) * 8) * C::PL + (lane >> 3 & 1) * 8;
            // with 8 columns per warp one ldmatrix brings both 16-token steps
            constexpr bool kPair = KW >= 16;
            const bf16 *b = tile_b(s & kMask) + (bw * TW + (kPair ? lane & 15 : lane)) * C::PK + kw + (kPair ? (lane >> 4) * 8 : 0);
            uint32_t fb[4];
            if (!kPair) ldsm4_trans(fb, b);
#pragma unroll
            for (int ks = 0; ks < TW / 16; ++ks) {
                uint32_t fa[LS / 16][4];
#pragma unroll
                for (int mt = 0; mt < LS / 16; ++mt) ldsm4_trans(fa[mt], a + ks * 16 * C::PL + mt * 16);
                if constexpr (kPair) {
#pragma unroll
                    for (int np = 0; np < KW / 16; ++np) {
                        ldsm4_trans(fb, b + ks * 16 * C::PK + np * 16);
#pragma unroll
                        for (int mt = 0; mt < LS / 16; ++mt) {
                            mma16816(acc[mt][2 * np], fa[mt], fb[0], fb[1]);
                            mma16816(acc[mt][2 * np + 1], fa[mt], fb[2], fb[3]);
                        }
                    }
                } else {
#pragma unroll
                    for (int mt = 0; mt < LS / 16; ++mt) mma16816(acc[mt][0], fa[mt], fb[2 * ks], fb[2 * ks + 1]);
                }
            }
        } else {
            const float *a = tile_a(s & kMask) + bw * C::kBlockL + (lane >> 3) * RL, *b = tile_b(s & kMask) + bw * C::kBlockK + kw + (lane & 7) * VK;
#pragma unroll 4
            for (int t = 0; t < TW; ++t) {
                if (C::KC > 0 && t == TW / 2 && mine == 1 && s + 1 < s1) load(s + 1);
                float fa[RL], fb[RK];
#pragma unroll
                for (int i = 0; i < RL; i += 4) *reinterpret_cast<float4 *>(fa + i) = *reinterpret_cast<const float4 *>(a + t * C::PL + i);
#pragma unroll
                for (int i = 0; i < RK; i += VK) {
                    if constexpr (VK == 4) *reinterpret_cast<float4 *>(fb + i) = *reinterpret_cast<const float4 *>(b + t * C::PK + 8 * i);
                    else                   *reinterpret_cast<float2 *>(fb + i) = *reinterpret_cast<const float2 *>(b + t * C::PK + 8 * i);
                }
#pragma unroll
                for (int i = 0; i < RL; ++i)
#pragma unroll
                    for (int k = 0; k < RK; ++k) acc[i][k][0] = fmaf(fa[i], fb[k], acc[i][k][0]);
            }
        }
        if (!early && s + 1 < s1) {
            if (C::kSteps == 1) __syncthreads();
            load(s + 1);
        }
    }
    if constexpr (C::kBf) {
        const int g = lane >> 2, q = lane & 3;
#pragma unroll
        for (int mt = 0; mt < LS / 16; ++mt)
#pragma unroll
            for (int nt = 0; nt < KW / 8; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 *d = reinterpret_cast<float2 *>(dst + (mt * 16 + g + 8 * h) * M + nt * 8 + 2 * q);
                    float2 r = make_float2(acc[mt][nt][2 * h], acc[mt][nt][2 * h + 1]);
                    if (add) { const float2 o = *d; r.x += o.x; r.y += o.y; }
                    *d = r;
                }
    } else {
#pragma unroll
        for (int i = 0; i < RL; ++i)
#pragma unroll
            for (int k = 0; k < RK; k += VK) {
                float *d = dst + ((lane >> 3) * RL + i) * M + (lane & 7) * VK + 8 * k;
                if constexpr (VK == 4) {
                    float4 r = make_float4(acc[i][k][0], acc[i][k + 1][0], acc[i][k + 2][0], acc[i][k + 3][0]);
                    if (add) { const float4 o = *reinterpret_cast<float4 *>(d); r.x += o.x; r.y += o.y; r.z += o.z; r.w += o.w; }
                    *reinterpret_cast<float4 *>(d) = r;
                } else {
                    float2 r = make_float2(acc[i][k][0], acc[i][k + 1][0]);
                    if (add) { const float2 o = *reinterpret_cast<float2 *>(d); r.x += o.x; r.y += o.y; }
                    *reinterpret_cast<float2 *>(d) = r;
                }
            }
    }
}

// ---------------------------------------------------------------- sums
constexpr int kReducePer = 1024;                       // elements of a reduce unit
__device__ __forceinline__ void reduce_unit(const Op &op, int unit)
{
    const long long i = (long long)unit * kReducePer + threadIdx.x * 4;
    if (threadIdx.x * 4 >= kReducePer || i >= op.count) return;
    float4 s = op.accumulate ? *reinterpret_cast<const float4 *>(op.sums + i) : make_float4(0, 0, 0, 0);
#pragma unroll 8
    for (int p = 0; p < op.splits; ++p) {
        const float4 v = *reinterpret_cast<const float4 *>(op.parts + p * op.count + i);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    *reinterpret_cast<float4 *>(op.sums + i) = s;
}

constexpr int kColsumCols = 64;                        // columns of a column-sum unit
template <typename C> __device__ __forceinline__ void colsum_unit(const Op &op, int unit, int tokens, unsigned char *smem)
{
    typedef typename C::T T;
    constexpr int N = C::M * C::M, V = 16 / (int)sizeof(T), kLanes = kColsumCols / V, kRows = C::kThreads / kLanes;
    const int cl = threadIdx.x % kLanes, r = threadIdx.x / kLanes;
    const T *src = static_cast<const T *>(op.in.p) + unit * kColsumCols + cl * V;
    float s[V] = {};
#pragma unroll 4
    for (int t = r; t < tokens; t += kRows) {
        const uint4 raw = *reinterpret_cast<const uint4 *>(src + (size_t)t * N);
#pragma unroll
        for (int e = 0; e < V; ++e) s[e] += elem<T>::load(reinterpret_cast<const T *>(&raw) + e);
    }
    float *red = reinterpret_cast<float *>(smem);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < V; ++e) red[r * kColsumCols + cl * V + e] = s[e];
    // pairwise: a chain over the rows would round a short sum more often than one over its tokens
#pragma unroll 1
    for (int half = kRows / 2; half > 0; half /= 2) {
        __syncthreads();
        for (int i = threadIdx.x; i < half * kColsumCols; i += C::kThreads) red[i] += red[i + half * kColsumCols];
    }
    __syncthreads();
    if (threadIdx.x < kColsumCols) {
        float *d = op.sums + unit * kColsumCols + threadIdx.x;
        *d = op.accumulate ? *d + red[threadIdx.x] : red[threadIdx.x];
    }
}

// Out of line beside products that need every register (fp32 m = 64, 2048 tokens: backward 283 -> 264 us).
template <typename C> __device__ __noinline__ void reduce_far(const Op &op, int unit) { reduce_unit(op, unit); }
template <typename C> __device__ __noinline__ void colsum_far(const Op &op, int unit, int tokens, unsigned char *smem) { colsum_unit<C>(op, unit, tokens, smem); }

// ---------------------------------------------------------------- the launch
struct Plan {                                          // shares of the CTAs, worked out on the host
    int units[kMaxOps], shift[kMaxOps];                // of an operation: units, and log2 of the weight of one
    long long share[kMaxOps], rest[kMaxOps];           // of a phase: total weight / and mod the number of CTAs
};

// Every CTA of the grid has arrived: all are resident (cooperative launch).  Bounded like every wait of the library.
__device__ __forceinline__ bool grid_barrier(unsigned *status, unsigned target, volatile int *dead)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(status + kBarrierWord, 1u);
        unsigned long long t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(status + kBarrierWord) : "memory");
            if (v >= target) break;
            if ((spin & 1023) == 1023) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                const unsigned us = reinterpret_cast<volatile unsigned *>(status)[1];
                if (now - t0 > (us ? us * 1000ull : 1000000000ull)) {
                    *dead = 1;
                    atomicCAS(status, 0u, kErrGridWait);
                    break;
                }
            }
        }
    }
    __syncthreads();
    return *dead == 0;
}

template <typename C>
__global__ void __launch_bounds__(C::kThreads, C::kCtas) units_kernel(const __grid_constant__ Params p, const __grid_constant__ Plan plan)
{
    constexpr int M = C::M;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int dead;
    if (threadIdx.x == 0) dead = 0;
    const int tiles = (int)((p.tokens + C::TT - 1) / C::TT);
    const int bid = blockIdx.x;
    int held_op = -1, held_at = -1;                    // whose weights are in shared memory

    // calls f(op, first unit, end) for this CTA's share of the operations of a phase, until f returns false
    auto share = [&](int phase, auto f) {
        const long long lo = bid * plan.share[phase] + min((long long)bid, plan.rest[phase]);
        const long long hi = lo + plan.share[phase] + (bid < plan.rest[phase]);
        long long base = 0;
        for (int o = 0; o < p.n_ops; ++o) {
            if (p.op[o].phase != phase) continue;
            const int sh = plan.shift[o];
            const long long w = 1ll << sh, n = plan.units[o];
            long long i0 = lo > base ? (lo - base + w - 1) >> sh : 0, i1 = hi > base ? (hi - base + w - 1) >> sh : 0;
            if (i0 > n) i0 = n;
            if (i1 > n) i1 = n;
            base += n << sh;
            if (i0 < i1 && !f(o, (int)i0, (int)i1)) return;
        }
    };

    for (int phase = 0; phase < p.n_phases; ++phase) {
        share(phase, [&](int o, int i0, int i1) {
            const Op &op = p.op[o];
            if (op.kind == kStage) {
                if (held_op != o) held_at = -1;
                if constexpr (C::KC > 0) stage_units_chunked<C>(op, i0, i1, tiles, p.tokens, smem);
                else                     stage_units<C>(op, i0, i1, tiles, p.tokens, smem, held_at);
                held_op = o;
                return true;
            }
            for (int i = i0; i < i1; ++i) {
                if (op.kind == kWgrad) {
                    constexpr int kL = M / C::LS, kK = M / C::KS;
                    wgrad_unit<C>(op, i / (kL * kK) % (M / 8) * 8, i / kK % kL * C::LS, i % kK * C::KS, i / (kL * kK * (M / 8)), p.tokens, smem);
                    held_op = -1;
                } else if (op.kind == kReduce) {
                    if constexpr (M > 16) reduce_far<C>(op, i);
                    else                  reduce_unit(op, i);
                } else {
                    if constexpr (M > 16) colsum_far<C>(op, i, p.tokens, smem);
                    else                  colsum_unit<C>(op, i, p.tokens, smem);
                    held_op = -1;
                }
            }
            return true;
        });
        if (phase + 1 == p.n_phases) break;
        // the weights of the next phase do not depend on this one: fetched while the barrier is waited for
        if constexpr (C::KC == 0) share(phase + 1, [&](int o, int i0, int) {
            if (p.op[o].kind == kStage) {
                const int at = i0 / tiles;
                if (held_op != o || held_at != at) {
                    __syncthreads();
                    load_weights<C>(reinterpret_cast<typename C::T *>(smem + C::kWAt), p.op[o].w, p.op[o].trans, at / (M / C::ES) * 8,
                                    at % (M / C::ES) * C::ES);
                    held_op = o;
                    held_at = at;
                }
            }
            return false;
        });
        if (!grid_barrier(p.status, (unsigned)(phase + 1) * gridDim.x, &dead)) break;
    }
    cp_async_wait();                                   // nothing in flight when the CTA exits, also after a timeout
    if (threadIdx.x == 0 && p.n_phases > 1 && dead == 0) {
        if (atomicAdd(p.status + kDoneWord, 1u) == gridDim.x - 1) {     // the last to leave puts the counters back to zero
            p.status[kBarrierWord] = 0;
            p.status[kDoneWord] = 0;
        }
    }
}

}  // namespace units
}  // namespace monarch
