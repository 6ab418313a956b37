// m = 32 (n = 1024), bf16: forward and backward with every intermediate on one SM.
//
// The weights of one stage are 64 KB: held as MMA operands in the registers of one CTA's 16 warps (two blocks per warp,
// 32 registers per stage) they are read once per launch, and shared memory is left to the token tiles.  A tile is 16
// tokens (32 KB per tensor), brought and taken by TMA.  Warp MMAs (m16n8k16): one stage is 2 GFLOP at 16384 tokens,
// 4 us of their rate, while the path is bound by HBM (10.3 us) - tcgen05 needs M = 64 rows of tokens or outputs per
// instruction, and its form of this kernel was bound by the issue of 128 such instructions per 64 tokens (29 us).
//
// The weights are the A operand (rows = outputs), the tokens are N, so every result fragment has tokens innermost and
// every permutation of Section 3.3 is a choice of where stmatrix puts a row of 8 tokens:
//   T tile  x, y, dy, dx in shared memory: [16 boxes of 64 columns][16 tokens][128 bytes], 16-byte chunks XORed with t % 8
//           (TMA's 128-byte swizzle)
//   E tile  a tensor by blocks: [block b][8-token half][row c of the block] chunks of 8 tokens, XORed with b % 8
//   forward:   u = R_k x_k  (B = T tile by ldmatrix)        -> E tile [j][k]:  row j of block k goes to block j (the P^T)
//              w = L_j u_j  (B = E tile by ldmatrix.trans)  -> E tile [j][l], in place: a warp overwrites its own blocks
//              y            E tile [j][l] -> T tile, 8 x 8 transposes by ldmatrix.trans / stmatrix (the outer P)
//   backward:  z = P dy     T tile -> E tile [j][l];   du = L_j^T z_j -> E tile [k][j];   dx = R_k^T du_k -> T tile
//              dL_j = sum_t z_j u_j^T, dR_k = sum_t du_k x_k^T: tokens are the contraction, both operands as they lie
// Shared memory moves 16 to 18 KB per token at 128 bytes per clock, no access has a bank conflict.
// Measured, back to back: forward 16384 tokens 29.2 -> 15.5 us (3.4 of it when the weights came to be loaded by TMA), 1000 tokens
// 14.5 -> 4.9; forward + backward 4999 tokens 103 -> 30.5, 16384 tokens 61 (the staged chain of nine
// launches took 219 as units and more as tcgen05 stages); feed-forward block 16384 tokens 167 -> 36.
//
// Backward CTAs are of three kinds, dL, dR and dx: the sums of one gradient are 128 KB of accumulators, half the
// registers of an SM, and a kind needs one or two sets of weights beside them.  u and du are recomputed by the kind that
// needs them (the MMAs are nearly free; the saved traffic is not).  Every CTA stores its sums, a second small launch adds
// them in a fixed order.
#include "mma_tiles.cuh"

namespace monarch {
namespace tc {
namespace {

constexpr int kM = 32, kN = kM * kM, kTok = 16, kWarps = 16, kThreads = kWarps * 32;
constexpr int kTile = kTok * kN * 2;                     // bytes of a T or E tile
constexpr int kSlots = 5, kSmemBytes = (kSlots + 2) * kTile + 1024;
constexpr int kKinds = 3, kDL = 0, kDR = 1, kDX = 2;
constexpr int kMaxParts = 50;                            // CTAs of a kind: a third of the chip

// chunk c (8 columns) of token t in a T tile; chunk (half h, row c) of block b in an E tile
__device__ __forceinline__ uint32_t t_at(uint32_t base, int box, int t, int c) { return base + box * (kTok * 128) + t * 128 + ((c ^ (t & 7)) << 4); }
__device__ __forceinline__ uint32_t e_at(uint32_t base, int b, int h, int c) { return base + b * 1024 + (((h * 32 + c) ^ (b & 7)) << 4); }

// chunk c of row r of block b of the weights
__device__ __forceinline__ uint32_t w_at(uint32_t base, int b, int r, int c)
{
    const int pair = b * (kM / 2) + (r >> 1);
    return base + pair * 128 + ((((r & 1) * 4 + c) ^ (pair & 7)) << 4);
}

// Operand A of a warp's two blocks: rows = outputs, [block][16 rows][16 columns of the contraction]
struct Weights {
    uint32_t a[2][2][2][4];
    // from the 32 blocks in shared memory, two rows of a block in 128 swizzled bytes
    __device__ __forceinline__ void load(uint32_t W, bool trans)
    {
        const Lane ln;
#pragma unroll
        for (int blk = 0; blk < 2; ++blk)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const int row = mt * 16 + (ln.m & 1) * 8, col = ks * 16 + (ln.m >> 1) * 8;       // of the 8 x 8 piece
                    if (trans) ldm4t(a[blk][mt][ks], w_at(W, ln.warp * 2 + blk, col + ln.r, row >> 3));
                    else       ldm4(a[blk][mt][ks], w_at(W, ln.warp * 2 + blk, row + ln.r, col >> 3));
                }
    }
    // acc = blk's rows times the operand b (both 16-column steps)
    __device__ __forceinline__ void times(int blk, const uint32_t (&b)[4], float (&acc)[2][4]) const
    {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            acc[mt][0] = acc[mt][1] = acc[mt][2] = acc[mt][3] = 0.0f;
            mma(acc[mt], a[blk][mt][0], b[0], b[1]);
            mma(acc[mt], a[blk][mt][1], b[2], b[3]);
        }
    }
};
__device__ __forceinline__ void pack_rows(const float (&acc)[2][4], uint32_t (&o)[4])       // the 8 x 8 pieces of 32 rows x 8 tokens
{
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        o[2 * mt] = pack_bf16(acc[mt][0], acc[mt][1]);
        o[2 * mt + 1] = pack_bf16(acc[mt][2], acc[mt][3]);
    }
}

// The operands of a stage are loaded together, ahead of its products.
struct Operands {
    uint32_t b[2][2][4];                                 // [block][8-token half]
    __device__ __forceinline__ void from_t(uint32_t T)
    {
        const Lane ln;
#pragma unroll
        for (int i = 0; i < 4; ++i) ldm4(b[i >> 1][i & 1], t_at(T, ln.warp, (i & 1) * 8 + ln.r, (i >> 1) * 4 + ln.m));
    }
    __device__ __forceinline__ void from_e(uint32_t E)   // rows of the warp's own blocks
    {
        const Lane ln;
#pragma unroll
        for (int i = 0; i < 4; ++i) ldm4t(b[i >> 1][i & 1], e_at(E, ln.warp * 2 + (i >> 1), i & 1, ln.m * 8 + ln.r));
    }
};
// E[row][own block] = W_block operand: row c of the result of block b becomes row b of block c
__device__ __forceinline__ void stage_to_e(const Weights &w, const Operands &in, uint32_t E)
{
    const Lane ln;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t o[4];
        float acc[2][4];
        w.times(i >> 1, in.b[i >> 1][i & 1], acc);
        pack_rows(acc, o);
        stm4(e_at(E, ln.m * 8 + ln.r, i & 1, ln.warp * 2 + (i >> 1)), o);
    }
}
// E[block][row] -> T (the outer P) and back; a warp takes the columns of one box
__device__ __forceinline__ void e_to_t(uint32_t E, uint32_t T)
{
    const Lane ln;
    uint32_t v[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) ldm4t(v[n], e_at(E, ln.m * 8 + ln.r, n >> 1, ln.warp * 2 + (n & 1)));
#pragma unroll
    for (int n = 0; n < 4; ++n) stm4(t_at(T, ln.warp, (n >> 1) * 8 + ln.r, (n & 1) * 4 + ln.m), v[n]);
}
__device__ __forceinline__ void t_to_e(uint32_t T, uint32_t E)
{
    const Lane ln;
    uint32_t v[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) ldm4t(v[n], t_at(T, ln.warp, (n >> 1) * 8 + ln.r, (n & 1) * 4 + ln.m));
#pragma unroll
    for (int n = 0; n < 4; ++n) stm4(e_at(E, ln.m * 8 + ln.r, n >> 1, ln.warp * 2 + (n & 1)), v[n]);
}

struct Params {
    unsigned *status;
    const __nv_bfloat16 *bias;
    float *parts;                // backward: [kDL, kDR][ranks][32][32][32]
    int tiles, gelu, ranks;
    int follows;                 // forward: behind another launch of the same call
    int skip;                    // test aid: one of CTA 0's first tiles, never loaded; -1: none
    __device__ __forceinline__ bool skips(int item) const { return blockIdx.x == 0 && item == skip; }
    int first[kKinds + 1];       // backward: CTAs of a kind start here
};

// Ring of T tiles filled by one thread, which waits for every tile like the others
struct Ring {
    uint32_t base, bars;
    unsigned *status;
    volatile int *dead;
    int loads;                                           // tiles to load: none any more once a wait of this thread has run out
    __device__ __forceinline__ uint32_t slot(int item) const { return base + (item % kSlots) * kTile; }
    __device__ __forceinline__ void load(int item, const CUtensorMap *m, int tile) const
    {
        const uint32_t bar = bars + (item % kSlots) * 8;
        mbar_expect_tx(bar, kTile);
        tma_load_3d(slot(item), m, 0, tile * kTok, 0, bar);
    }
    // A wait that runs out leaves `dead` set and garbage in the tile; the loops still run to their end, every later wait returns at
    // once.  The slot may be asked for again although its copy is still under way, and arming a barrier in the middle of its phase
    // is undefined: nothing is loaded any more.
    __device__ __forceinline__ uint32_t wait(int item)
    {
        if (!mbar_wait(bars + (item % kSlots) * 8, (item / kSlots) & 1, status, dead, kErrTmaWait)) loads = 0;
        return slot(item);
    }
};

struct Shared {
    uint64_t bars[kSlots], w_full;
    int dead;
};
constexpr int kWeightBytes = kM * kM * kM * 2;           // of one factor: two tiles
// The weights of a CTA come by TMA through shared memory that the first tiles do not need yet, and go to registers by ldmatrix.
// (Fetched by the warps in 4-byte pieces of the operand layout they took 4 us: eight lines per load.)
__device__ __forceinline__ void load_weights(uint32_t to, const CUtensorMap *m, Shared &s)
{
    for (int i = 0; i < 2; ++i) tma_load_2d(to + i * (kWeightBytes / 2), m, 0, i * 256, smem_u32(&s.w_full));
}
__device__ __forceinline__ void init(Shared &s)
{
    if (threadIdx.x == 0) {
        for (int i = 0; i < kSlots; ++i) mbar_init(smem_u32(&s.bars[i]), 1);
        mbar_init(smem_u32(&s.w_full), 1);
        fence_mbar_init();
        s.dead = 0;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- forward
// Per tile two barriers: [w(i) from u(i), u(i + 1) from x] [y(i)].  ACT: y = GELU(M x + bias), or without the GELU.
template <bool ACT>
__global__ void __launch_bounds__(kThreads, 1)
fused_fwd_m32_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_L,
                     const __grid_constant__ CUtensorMap tm_R, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    Ring ring = {base, smem_u32(sh.bars), p.status, &sh.dead, 0};
    const uint32_t E[2] = {base + kSlots * kTile, base + (kSlots + 1) * kTile};
    init(sh);
    const int first = blockIdx.x, step = gridDim.x, count = (p.tiles - first + step - 1) / step;
    ring.loads = count;
    const int warp = threadIdx.x >> 5;
    Weights wr, wl;
    auto weights = [&] {
        mbar_expect_tx(smem_u32(&sh.w_full), 2 * kWeightBytes);
        load_weights(ring.slot(3), &tm_R, sh);
        load_weights(E[0], &tm_L, sh);
    };
    // The second pass of a feed-forward block asks for its weights before it waits for the first one: that one lets its followers
    // begin only after its own wait, so what ran before the call has finished.
    if (p.follows && threadIdx.x == 0) weights();
    depend_wait();
    depend_launch();
    if (threadIdx.x == 0) {
        if (!p.follows) weights();
        for (int i = 0; i < 3 && i < count; ++i)
            if (!p.skips(i)) ring.load(i, &tm_x, first + i * step);
    }
    float bias[2][4];
    if (ACT)
#pragma unroll
        for (int i = 0; i < 8; ++i)                      // row l = 8 (i % 4) + lane / 4 of block j
            bias[i >> 2][i & 3] = __bfloat162float(p.bias[((i & 3) * 8 + ((threadIdx.x & 31) >> 2)) * kM + warp * 2 + (i >> 2)]);

    const Lane ln;
    Operands in;
    mbar_wait(smem_u32(&sh.w_full), 0, p.status, &sh.dead, kErrTmaWait);
    wr.load(ring.slot(3), false);
    wl.load(E[0], false);
    in.from_t(ring.wait(0));
    __syncthreads();                                     // every warp has its weights
    stage_to_e(wr, in, E[0]);
    for (int i = 0; i < count; ++i) {
        const uint32_t e = E[i & 1];
        __syncthreads();                                 // u(i) and y(i - 1) are complete
        if (threadIdx.x == 0) {
            if (i > 0) {
                tma_store_3d(&tm_y, ring.slot(i - 1), 0, (first + (i - 1) * step) * kTok, 0);
                tma_store_commit();
            }
            if (i + 3 < ring.loads) {
                tma_store_wait_read<1>();                // y(i - 2) has left its slot
                ring.load(i + 3, &tm_x, first + (i + 3) * step);
            }
        }
        const bool more = i + 1 < count;
        in.from_e(e);
        Operands nx;
        if (more) nx.from_t(ring.wait(i + 1));
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            uint32_t o[4];
            float acc[2][4];
            wl.times(v >> 1, in.b[v >> 1][v & 1], acc);
            if (ACT)
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    acc[k >> 2][k & 3] += bias[v >> 1][k >> 1];
                    acc[k >> 2][(k & 3) + 1] += bias[v >> 1][k >> 1];
                    if (p.gelu) gelu_fast2(acc[k >> 2][k & 3], acc[k >> 2][(k & 3) + 1]);
                }
            pack_rows(acc, o);
            stm4(e_at(e, warp * 2 + (v >> 1), v & 1, ln.m * 8 + ln.r), o);
        }
        if (more) stage_to_e(wr, nx, E[(i + 1) & 1]);
        __syncthreads();                                 // w(i) is complete; x(i) has been read by everyone
        e_to_t(e, ring.slot(i));
        fence_proxy_async_smem();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        tma_store_3d(&tm_y, ring.slot(count - 1), 0, (first + (count - 1) * step) * kTok, 0);
        tma_store_commit();
        tma_store_wait_all<0>();
    }
    let_copies_land(&sh.dead);
}

// ---------------------------------------------------------------- backward
// sums[block][32 rows][32 columns] += A (rows, tokens) B (tokens, columns) of the warp's two blocks; A rows are rows of an
// E tile; B likewise, or columns of a T tile
struct Sums {
    float v[2][2][4][4];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i >> 5][i >> 4 & 1][i >> 2 & 3][i & 3] = 0.0f;
    }
    template <bool BT> __device__ __forceinline__ void add(uint32_t A, uint32_t B)
    {
        const Lane ln;
#pragma unroll
        for (int blk = 0; blk < 2; ++blk) {
            const int own = ln.warp * 2 + blk;
            uint32_t a[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) ldm4(a[mt], e_at(A, own, ln.m >> 1, mt * 16 + (ln.m & 1) * 8 + ln.r));
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                uint32_t b[4];
                const int col = np * 2 + (ln.m >> 1), half = ln.m & 1;
                if (BT) ldm4t(b, t_at(B, ln.warp, half * 8 + ln.r, blk * 4 + col));
                else    ldm4(b, e_at(B, own, half, col * 8 + ln.r));
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    mma(v[blk][mt][2 * np], a[mt], b[0], b[1]);
                    mma(v[blk][mt][2 * np + 1], a[mt], b[2], b[3]);
                }
            }
        }
    }
    __device__ __forceinline__ void store(float *to) const
    {
        const int warp = threadIdx.x >> 5, g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
#pragma unroll
        for (int blk = 0; blk < 2; ++blk)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<float2 *>(to + (size_t)(warp * 2 + blk) * kM * kM + (mt * 16 + g + 8 * h) * kM + nt * 8 + 2 * q) =
                            make_float2(v[blk][mt][nt][2 * h], v[blk][mt][nt][2 * h + 1]);
    }
};

__global__ void __launch_bounds__(kThreads, 1)
fused_bwd_m32_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dy,
                     const __grid_constant__ CUtensorMap tm_dx, const __grid_constant__ CUtensorMap tm_L, const __grid_constant__ CUtensorMap tm_R,
                     const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    Ring ring = {base, smem_u32(sh.bars), p.status, &sh.dead, 0};
    const uint32_t V = base + kSlots * kTile, U = V + kTile;
    init(sh);
    const int b = blockIdx.x, kind = b < p.first[1] ? kDL : b < p.first[2] ? kDR : kDX;
    const int first = b - p.first[kind], step = p.first[kind + 1] - p.first[kind], count = (p.tiles - first + step - 1) / step;
    ring.loads = kind == kDX ? count : 2 * count;
    const int warp = threadIdx.x >> 5;

    if (kind == kDX) {
        // per tile [du(i) from z(i)] [dx(i), z(i + 1)]
        Weights wl, wr;
        depend_wait();
        depend_launch();
        if (threadIdx.x == 0) {
            mbar_expect_tx(smem_u32(&sh.w_full), 2 * kWeightBytes);
            load_weights(ring.slot(3), &tm_L, sh);
            load_weights(V, &tm_R, sh);
            for (int i = 0; i < 3 && i < count; ++i)
                if (!p.skips(i)) ring.load(i, &tm_dy, first + i * step);
        }
        mbar_wait(smem_u32(&sh.w_full), 0, p.status, &sh.dead, kErrTmaWait);
        wl.load(ring.slot(3), true);
        wr.load(V, true);
        __syncthreads();                                 // every warp has its weights
        const Lane ln;
        Operands in;
        t_to_e(ring.wait(0), V);
        for (int i = 0; i < count; ++i) {
            __syncthreads();                             // z(i) and dx(i - 1) are complete
            if (threadIdx.x == 0) {
                if (i > 0) {
                    tma_store_3d(&tm_dx, ring.slot(i - 1), 0, (first + (i - 1) * step) * kTok, 0);
                    tma_store_commit();
                }
                if (i + 3 < ring.loads) {
                    tma_store_wait_read<1>();
                    ring.load(i + 3, &tm_dy, first + (i + 3) * step);
                }
            }
            in.from_e(V);
            stage_to_e(wl, in, U);
            __syncthreads();                             // du(i) is complete, z(i) has been read
            in.from_e(U);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                uint32_t o[4];
                float acc[2][4];
                wr.times(v >> 1, in.b[v >> 1][v & 1], acc);
                pack_rows(acc, o);
                stm4t(t_at(ring.slot(i), warp, (v & 1) * 8 + ln.r, (v >> 1) * 4 + ln.m), o);
            }
            fence_proxy_async_smem();
            if (i + 1 < count) t_to_e(ring.wait(i + 1), V);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            tma_store_3d(&tm_dx, ring.slot(count - 1), 0, (first + (count - 1) * step) * kTok, 0);
            tma_store_commit();
            tma_store_wait_all<0>();
        }
        let_copies_land(&sh.dead);
        return;
    }
    // items of the ring: dy(i) = 2 i, x(i) = 2 i + 1
    int next = 0;
    auto load_to = [&](int last) {
        for (; next <= last && next < ring.loads; ++next)
            if (!p.skips(next)) ring.load(next, next & 1 ? &tm_x : &tm_dy, first + (next >> 1) * step);
    };
    Weights w;
    Operands in;
    Sums sums;
    sums.clear();
    depend_wait();
    depend_launch();
    if (threadIdx.x == 0) {
        mbar_expect_tx(smem_u32(&sh.w_full), kWeightBytes);
        load_weights(V, kind == kDL ? &tm_R : &tm_L, sh);
        load_to(kSlots - 1);
    }
    mbar_wait(smem_u32(&sh.w_full), 0, p.status, &sh.dead, kErrTmaWait);
    w.load(V, kind != kDL);
    __syncthreads();                                     // every warp has its weights
    if (kind == kDL) {
        // per tile [sums from z(i), u(i)] [z(i + 1), u(i + 1)]
        t_to_e(ring.wait(0), V);
        in.from_t(ring.wait(1));
        stage_to_e(w, in, U);
        for (int i = 0; i < count; ++i) {
            __syncthreads();
            if (threadIdx.x == 0) load_to(2 * i + 1 + kSlots);
            sums.add<false>(V, U);
            __syncthreads();
            if (i + 1 < count) {
                t_to_e(ring.wait(2 * i + 2), V);
                in.from_t(ring.wait(2 * i + 3));
                stage_to_e(w, in, U);
            }
        }
    } else {
        // per tile [du(i) from z(i)] [sums from du(i), x(i); z(i + 1)]
        t_to_e(ring.wait(0), V);
        for (int i = 0; i < count; ++i) {
            __syncthreads();                             // z(i) is complete; x(i - 1) has been read
            if (threadIdx.x == 0) load_to(2 * i + kSlots);
            in.from_e(V);
            stage_to_e(w, in, U);
            const uint32_t x = ring.wait(2 * i + 1);
            __syncthreads();
            sums.add<true>(U, x);
            if (i + 1 < count) t_to_e(ring.wait(2 * i + 2), V);
        }
    }
    sums.store(p.parts + ((size_t)kind * p.ranks + first) * kM * kM * kM);
    let_copies_land(&sh.dead);
}

// grads = (accumulate ? grads : 0) + the parts, in order; 32 groups of 4 elements and 8 ranges of parts per CTA
__global__ void __launch_bounds__(256)
add_parts_m32_kernel(const float *__restrict__ parts, float *__restrict__ dL, float *__restrict__ dR, int n, int accumulate)
{
    __shared__ float4 red[8][32];
    constexpr int kElems = kM * kM * kM, kPer = 32 * 4;
    const int kind = blockIdx.x / (kElems / kPer), at = blockIdx.x % (kElems / kPer) * kPer + (threadIdx.x & 31) * 4;
    const int range = threadIdx.x >> 5;
    const float *src = parts + (size_t)kind * n * kElems + at;
    float *dst = (kind == kDL ? dL : dR) + at;
    const int per = (n + 7) / 8;
    float4 s = make_float4(0, 0, 0, 0);
    depend_wait();
#pragma unroll 7
    for (int i = range * per; i < (range + 1) * per && i < n; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(src + (size_t)i * kElems);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    red[range][threadIdx.x & 31] = s;
    __syncthreads();
    if (range == 0) {
        if (accumulate) {
            const float4 o = *reinterpret_cast<const float4 *>(dst);
            s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
        }
#pragma unroll
        for (int i = 1; i < 8; ++i) {
            const float4 v = red[i][threadIdx.x];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4 *>(dst) = s;
    }
}

// [tokens][1024] as boxes of 64 columns: one copy of 64 x 16 tokens x 16 boxes is a T tile
int map_tile(CUtensorMap *m, const void *p, int64_t tokens)
{
    const uint64_t dims[3] = {64, (uint64_t)tokens, 16}, strides[2] = {kN * 2, 128};
    const uint32_t box[3] = {64, kTok, 16};
    return encode_tmap_nd(m, p, 2, 3, dims, strides, box, 128);
}

// the blocks of a factor as rows of 128 bytes
int map_weights(CUtensorMap *m, const void *W) { return encode_tmap_2d(m, W, kM * kM * kM / 64, 64, 128, 256, 64, 128); }

// bias null: y = M x
int launch_fwd_m32(const void *x, const void *L, const void *R, const void *bias, int gelu, void *y, int64_t tokens, void *ws,
                   int follows, cudaStream_t s)
{
    if (tokens == 0) return MONARCH_OK;
    if (tokens > 0x7fffffffLL - kTok) return MONARCH_ERR_UNSUPPORTED;
    CUtensorMap tm_x, tm_y, tm_L, tm_R;
    MONARCH_TRY(map_tile(&tm_x, x, tokens));
    MONARCH_TRY(map_tile(&tm_y, y, tokens));
    MONARCH_TRY(map_weights(&tm_L, L));
    MONARCH_TRY(map_weights(&tm_R, R));
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    auto kern = bias != nullptr ? fused_fwd_m32_kernel<true> : fused_fwd_m32_kernel<false>;
    Params p = {};
    p.skip = take_skipped_tile();
    p.status = (unsigned *)ws;
    p.bias = (const __nv_bfloat16 *)bias;
    p.gelu = gelu;
    p.follows = follows;
    p.tiles = (int)((tokens + kTok - 1) / kTok);
    return launch_serialized(kern, p.tiles < sms ? p.tiles : sms, kThreads, kSmemBytes, s, tm_x, tm_y, tm_L, tm_R, p);
}

}  // namespace
}  // namespace tc

// Workspace: only the status word is used.
int fused_fwd_m32(const void *x, const void *L, const void *R, void *y, int64_t tokens, void *ws, cudaStream_t s)
{
    return tc::launch_fwd_m32(x, L, R, nullptr, 0, y, tokens, ws, 0, s);
}

// The feed-forward block as two passes; workspace: status word, then h.
size_t fused_mlp_fwd_m32_workspace_bytes(int64_t tokens)
{
    return MONARCH_STATUS_BYTES + (((size_t)tokens * tc::kN * 2 + 255) & ~(size_t)255);
}
int fused_mlp_fwd_m32(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2,
                      void *y, int64_t tokens, void *ws, cudaStream_t s)
{
    void *h = (char *)ws + MONARCH_STATUS_BYTES;
    MONARCH_TRY(tc::launch_fwd_m32(x, L1, R1, b1, 1, h, tokens, ws, 0, s));
    return tc::launch_fwd_m32(h, L2, R2, b2, 0, y, tokens, ws, 1, s);
}

// Workspace: status word, then the sums of every CTA (64 KB are left out for the counters of the kernels that share it).
size_t fused_bwd_m32_workspace_bytes(int64_t tokens)
{
    const int64_t tiles = (tokens + tc::kTok - 1) / tc::kTok;
    return MONARCH_STATUS_BYTES + 65536 + (size_t)2 * (tiles < tc::kMaxParts ? tiles : tc::kMaxParts) * tc::kM * tc::kM * tc::kM * sizeof(float);
}
// dx null: gradients only; dL null: dx only
int fused_bwd_m32(const void *x, const void *dy, const void *L, const void *R, void *dx, float *dL, float *dR, int accumulate,
                  int64_t tokens, void *ws, cudaStream_t s)
{
    using namespace tc;
    if (tokens == 0) {
        if (dL != nullptr && !accumulate) {
            MONARCH_CUDA_TRY(cudaMemsetAsync(dL, 0, kM * kM * kM * sizeof(float), s));
            MONARCH_CUDA_TRY(cudaMemsetAsync(dR, 0, kM * kM * kM * sizeof(float), s));
        }
        return MONARCH_OK;
    }
    if (tokens > 0x7fffffffLL - kTok) return MONARCH_ERR_UNSUPPORTED;
    CUtensorMap tm_x, tm_dy, tm_dx, tm_L, tm_R;
    MONARCH_TRY(map_weights(&tm_L, L));
    MONARCH_TRY(map_weights(&tm_R, R));
    MONARCH_TRY(map_tile(&tm_dy, dy, tokens));
    MONARCH_TRY(map_tile(&tm_x, dL != nullptr ? x : dy, tokens));
    MONARCH_TRY(map_tile(&tm_dx, dx != nullptr ? dx : dy, tokens));
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    Params p = {};
    p.skip = take_skipped_tile();
    p.status = (unsigned *)ws;
    p.parts = (float *)((char *)ws + MONARCH_STATUS_BYTES + 65536);
    p.tiles = (int)((tokens + kTok - 1) / kTok);
    // The kinds cost the same per tile (256 KB of shared-memory traffic): equal shares, and the same share of a gradient
    // whether or not dx is asked for, so that its sums have the same bits.
    const int share = sms / kKinds < kMaxParts ? sms / kKinds : kMaxParts;
    const int most[kKinds] = {dL != nullptr ? share : 0, dL != nullptr ? share : 0, dx == nullptr ? 0 : dL != nullptr ? sms - 2 * share : sms};
    int n[kKinds];
    for (int k = 0; k < kKinds; ++k) {
        n[k] = most[k] < p.tiles ? most[k] : p.tiles;
        p.first[k + 1] = p.first[k] + n[k];
    }
    p.ranks = n[kDL];
    MONARCH_TRY(launch_serialized(fused_bwd_m32_kernel, p.first[kKinds], kThreads, kSmemBytes, s, tm_x, tm_dy, tm_dx, tm_L, tm_R, p));
    if (dL == nullptr) return MONARCH_OK;
    return launch_serialized(add_parts_m32_kernel, 2 * kM * kM * kM / 128, 256, 0, s, (const float *)p.parts, dL, dR, p.ranks, accumulate);
}

}  // namespace monarch
