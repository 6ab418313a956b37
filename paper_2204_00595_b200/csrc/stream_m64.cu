// m = 64 (n = 4096), bf16: forward, backward and feed-forward block as streaming launches, one per block-diagonal stage.
// Small forwards and blocks run on clusters of eight CTAs instead, one launch per multiply (further down).
//
// The weights of a stage are 512 KB, so an SM cannot hold both stages and every block of stage 2 needs a row of every block
// of stage 1: the intermediate has to cross SMs.  Each launch is one stage for all tokens: a CTA keeps the weights of its 16
// (backward: 8) blocks as warp-MMA operands in registers, read once, and streams 16-token tiles of just those blocks through
// shared memory by TMA.  Nothing waits for another CTA inside a launch.  Each launch walks the tiles in the opposite direction
// of the one before it: what that one wrote last is still in L2.  (Chunks of tokens whose intermediate stays there cost more in
// launches and last waves than they save: 4096 tokens a chunk, 194 us forward and backward at 8192 tokens, none 164.)
// The intermediates are stored as the next stage's operands lie in shared memory:
//   E tile  [tile of 16 tokens][8 consumer blocks][producer block p][8-token half][consumer c % 8] chunks of 8 tokens, the last
//           XORed with p % 8: 16 KB per 8 consumers; a consumer's blocks are one linear copy, a producer's 16 (8) blocks eight
//           of 4 (2) KB
//   T tile  natural rows of 64 columns, 128 bytes per token, 16-byte chunks XORed with t % 8 (TMA's 128-byte swizzle)
//   Y tile  [l][token][16 neighbouring columns j]: the 32-byte pieces of a permuted row (TMA's 32-byte swizzle)
// forward   x --T--> u_k = R_k x_k --E--> w_j = L_j u_j, in place in the E tile, transposed 8 x 8 to Y --> y
// backward  dy --(8 columns j)--> z_j, transposed to E; du_j = L_j^T z_j --E--> dx_k = R_k^T du_k --T--> dx
//           dL_j = sum_t z_j u_j^T beside du, dR_k = sum_t du_k x_k^T beside dx: tokens are the contraction, operands as they
//           lie; a CTA's sums are 128 KB of accumulators (half of its registers), stored once and added by a last launch in a
//           fixed order.
// A warp works on its own blocks and only the transposes look across, so warps run ahead of one another between mbarriers;
// the warps ask for tiles and send results away by turns, one tile behind their own work (a warp for that alone would cost
// every other one 32 of its 128 registers).  With a CTA barrier per tile instead, loads, MMAs and stores of a
// tile followed one another (2650 cycles per 32 KB tile and stage against 1030 of MMA and 1000 to 1500 of shared memory).
// The weights arrive by TMA as swizzled rows and go to registers by ldmatrix (1 us; fetched by the warps themselves in the
// 16-byte pieces of the operand layout they took 4).
#include "mma_tiles.cuh"

namespace monarch {
namespace tc {
namespace {

constexpr int kM = 64, kN = kM * kM, kTok = 16, kWarps = 16, kThreads = kWarps * 32;
constexpr int kRowBytes = 2 * 8 * 16;                    // a producer's 16 tokens for 8 consumers
constexpr int kGroupBytes = kM * kRowBytes;              // 8 consumers of an E tile: 16 KB
constexpr int kTileBytes = kM / 8 * kGroupBytes;         // an E tile: 128 KB
constexpr int kFwdBlocks = 16, kFwdGroups = kM / kFwdBlocks, kFwdTile = kTok * kFwdBlocks * kM * 2;   // 32 KB of any kind
constexpr int kBwdBlocks = 8, kBwdGroups = kM / kBwdBlocks, kBwdTile = kTok * kBwdBlocks * kM * 2;    // 16 KB
// shared memory in tiles: slots of the input ring, then V tiles (du), then staging tiles of the results.  The last four tiles
// hold the weights first.
constexpr int kFwdSlots = 4, kFwdStages = 3, kFwdSmem = (kFwdSlots + kFwdStages) * kFwdTile + 1024;
constexpr int kDuSlots = 8, kDuStages = 3, kDxSlots = 10, kDxStages = 4, kBwdSmem = 14 * kBwdTile + 1024;
constexpr int kMaxRanks = 19;                            // CTAs of a group in the backward launches (148 / 8, rounded up)
constexpr size_t kGradElems = (size_t)kM * kM * kM;

__device__ __forceinline__ uint32_t t_at(uint32_t base, int box, int t, int c) { return base + box * (kTok * 128) + t * 128 + ((c ^ (t & 7)) << 4); }
__device__ __forceinline__ uint32_t e_at(uint32_t base, int b, int h, int c) { return base + (b >> 3) * kGroupBytes + c * kRowBytes + h * 128 + (((b ^ c) & 7) << 4); }
// results for consumer block b from the CTA's block c of `blocks`, in a staging tile that leaves as eight linear pieces
__device__ __forceinline__ uint32_t out_at(uint32_t base, int blocks, int b, int h, int c) { return base + ((b >> 3) * blocks + c) * kRowBytes + h * 128 + (((b ^ c) & 7) << 4); }
// (of map_e) by the CTA's group of `blocks` producers
__device__ __forceinline__ void store_e(const CUtensorMap *m, int64_t tile, uint32_t from, int group, int blocks)
{
    tma_store_3d(m, from, 0, group * (blocks / 8), (int)tile * (kM / 8));
}

struct Params {
    unsigned *status;
    const __nv_bfloat16 *bias;
    const char *e_in, *u;        // E tiles that linear copies read
    char *e_out, *u_out;         // E tiles that linear copies write
    float *parts;                // [rank][64][64][64]
    int tiles;
    int last;                    // tiles - 1: from the last tile to the first; 0: from the first to the last
    int follows;                 // behind another launch of the same call: init()
    int skip;                    // test aid: one of CTA 0's first tiles, never loaded; -1: none
    __device__ __forceinline__ bool skips(int item) const { return blockIdx.x == 0 && item == skip; }
};

// Rows r0 .. r0 + 16 MT of one block, as operand A, from its 64 rows of 128 bytes in shared memory
template <int MT> struct Weights {
    uint32_t a[MT][4][4];
    __device__ __forceinline__ void load(uint32_t block, int r0, bool trans)
    {
        const Lane ln;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const int row = r0 + mt * 16 + (ln.m & 1) * 8, col = ks * 16 + (ln.m >> 1) * 8;      // of the 8 x 8 piece
                if (trans) ldm4t(a[mt][ks], block + (col + ln.r) * 128 + (((row >> 3) ^ ln.r) << 4));
                else       ldm4(a[mt][ks], block + (row + ln.r) * 128 + (((col >> 3) ^ ln.r) << 4));
            }
    }
    __device__ __forceinline__ void times(int mt, const uint32_t (&b)[2][4], float (&acc)[4]) const
    {
        acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) mma(acc, a[mt][ks], b[ks >> 1][(ks & 1) * 2], b[ks >> 1][(ks & 1) * 2 + 1]);
    }
};

struct Ring {
    uint32_t base, bars;
    int slots, bytes;
    unsigned *status;
    volatile int *dead;
    int loads;                   // items to load: none any more once a wait of this thread has run out
    __device__ __forceinline__ uint32_t slot(int item) const { return base + (item % slots) * bytes; }
    __device__ __forceinline__ uint32_t expect(int item) const
    {
        mbar_expect_tx(bars + (item % slots) * 8, bytes);
        return bars + (item % slots) * 8;
    }
    __device__ __forceinline__ void load(int item, const CUtensorMap *m, int tile, int z, int x = 0) const
    {
        tma_load_3d(slot(item), m, x, tile * kTok, z, expect(item));
    }
    __device__ __forceinline__ void load_linear(int item, const char *from) const
    {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(slot(item)), "l"(from),
                     "r"(bytes), "r"(expect(item)) : "memory");
    }
    // A wait that runs out leaves `dead` set and garbage in the tile; the loops still run to their end, every later wait returns at
    // once.  The slot may be asked for again although its copy is still under way, and arming a barrier in the middle of its phase
    // is undefined: the thread loads nothing more (one whose own wait succeeded may: that phase is complete).
    __device__ __forceinline__ uint32_t wait(int item)
    {
        if (!mbar_wait(bars + (item % slots) * 8, (item / slots) & 1, status, dead, kErrTmaWait)) loads = 0;
        return slot(item);
    }
};
constexpr int kMaxSlots = 10, kMaxStages = 8;
struct Shared {
    uint64_t full[kMaxSlots], staged[kMaxStages], free_[kMaxStages];
    uint64_t across[kFwdSlots];          // tiles that the transposes read: every warp has written its part
    uint64_t w_full, w_read;
    int dead;
};
// Barriers of a CTA.  staged(i): the results of tile i are in staging tile i % stages, and every warp is done with its inputs.
struct Sync {
    Shared &s;
    unsigned *status;
    int stages, across_n;
    __device__ __forceinline__ bool wait(const uint64_t &bar, int phase, unsigned code) const
    {
        return mbar_wait(smem_u32(&bar), phase & 1, status, &s.dead, code);
    }
    __device__ __forceinline__ static void arrive(uint64_t &bar)             // one per warp
    {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(&bar));
    }
    __device__ __forceinline__ void wait_staging(int i) const                // staging tile i % stages may be written
    {
        if (i < stages) wait(s.w_read, 0, kErrSlotWait);
        else            wait(s.free_[i % stages], i / stages - 1, kErrSlotWait);
    }
    __device__ __forceinline__ void staged(int i) const
    {
        fence_proxy_async_smem();
        arrive(s.staged[i % stages]);
    }
    __device__ __forceinline__ void wait_staged(int i) const { wait(s.staged[i % stages], i / stages, kErrMmaWait); }
    __device__ __forceinline__ void across(int i) const { arrive(s.across[i % across_n]); }
    __device__ __forceinline__ void wait_across(int i) const { wait(s.across[i % across_n], i / across_n, kErrMmaWait); }
    // Tiles are passed on by turns, each by three warps while the others go on: after its own tile k, warp k - 1 sends tile k - 1
    // away, warp k + 7 has the tiles loaded whose slots that one's inputs leave free, and warp k - 2 frees the staging of tile
    // k - 2 (all mod 16; by one warp for all tiles this took 400 to 1500 cycles of every tile, and the others waited).
    template <typename Send, typename Load> __device__ __forceinline__ void pass_on(int k, Send send, Load load) const
    {
        if (k >= 1 && (turn(k - 1) || turn(k + 7))) {
            wait_staged(k - 1);
            if (turn(k - 1)) {
                send(k - 1);
                tma_store_commit();
                if (stages == 2) {                           // the next tile needs it
                    tma_store_wait_read<0>();
                    mbar_arrive(smem_u32(&s.free_[(k - 1) % stages]));
                }
            } else {
                load(k - 1);
            }
        }
        if (stages > 2 && k >= 2 && turn(k - 2)) {
            tma_store_wait_read<0>();
            mbar_arrive(smem_u32(&s.free_[(k - 2) % stages]));
        }
        __syncwarp();
    }
    template <typename Send> __device__ __forceinline__ void pass_last(int count, Send send) const
    {
        if (count > 0 && turn(count - 1)) {
            wait_staged(count - 1);
            send(count - 1);
            tma_store_commit();
        }
        tma_store_wait_all<0>();
        __syncwarp();
    }
    __device__ __forceinline__ static bool turn(int k) { return threadIdx.x == (k & (kWarps - 1)) * 32; }
    // `blocks` blocks of W from block `first` on, as [row][64 columns] with 128-byte swizzle
    __device__ __forceinline__ void load_weights(uint32_t to, const CUtensorMap *tm_w, int first, int blocks, int planes = 1) const
    {
        const uint32_t bar = smem_u32(&s.w_full);
        mbar_expect_tx(bar, planes * blocks * kM * 128);
        for (int c = 0; c < planes; ++c)
            for (int b = 0; b < blocks; b += 4) tma_load_2d(to + (c * blocks + b) * kM * 128, tm_w, 0, c * kN + (first + b) * kM, bar);
    }
    template <int MT> __device__ __forceinline__ void take_weights(Weights<MT> &w, uint32_t block, int r0, bool trans) const
    {
        wait(s.w_full, 0, kErrTmaWait);
        w.load(block, r0, trans);
        arrive(s.w_read);
    }
    __device__ __forceinline__ void leave() const { let_copies_land(&s.dead); }
};
// weights(): by one thread.  A launch behind another one of its call asks for them before it waits for that one, which lets its
// followers begin only after its own wait: what ran before the call has finished.
template <typename F> __device__ __forceinline__ void begin(int follows, F weights)
{
    if (follows && threadIdx.x == 0) weights();
    depend_wait();
    depend_launch();
    if (!follows && threadIdx.x == 0) weights();
}
template <typename F> __device__ __forceinline__ void init(Shared &s, int follows, F weights)
{
    if (threadIdx.x == 0) {
        for (uint64_t &b : s.full) mbar_init(smem_u32(&b), 1);
        for (uint64_t &b : s.staged) mbar_init(smem_u32(&b), kWarps);
        for (uint64_t &b : s.free_) mbar_init(smem_u32(&b), 1);
        for (uint64_t &b : s.across) mbar_init(smem_u32(&b), kWarps);
        mbar_init(smem_u32(&s.w_full), 1);
        mbar_init(smem_u32(&s.w_read), kWarps);
        fence_mbar_init();
        s.dead = 0;
    }
    __syncthreads();
    begin(follows, weights);
}
// CTA -> (group of blocks, rank among the CTAs of that group)
__device__ __forceinline__ int ranks_of(int groups, int group) { return ((int)gridDim.x - group + groups - 1) / groups; }

// Biases of the rows of a warp's block `own` that a lane has results of: 16 mt + lane / 4 and + 8, as bf16 pairs
struct Bias {
    uint32_t v[4];
    __device__ __forceinline__ void load(const __nv_bfloat16 *bias, int own)
    {
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) {
            const unsigned short *at = reinterpret_cast<const unsigned short *>(bias) + (mt * 16 + ((threadIdx.x & 31) >> 2)) * kM + own;
            v[mt] = __ldg(at) | (uint32_t)__ldg(at + 8 * kM) << 16;
        }
    }
    __device__ __forceinline__ void add(int mt, float (&acc)[4]) const
    {
        const float lo = __uint_as_float(v[mt] << 16), hi = __uint_as_float(v[mt] & 0xFFFF0000u);
        acc[0] += lo;
        acc[1] += lo;
        acc[2] += hi;
        acc[3] += hi;
    }
};
// ---------------------------------------------------------------- forward, stage 1: x -> u (E tiles)
// E_IN: from E tiles; ACT: u = GELU(. + bias).  The middle of a feed-forward block is E tiles on both sides: stage 2 of the first
// matrix and stage 1 of the second are this kernel too, and h needs no transposes (8192 tokens 103 -> 100 us, 32768 383 -> 375; the
// GELU alone is 20 of that: without one the same launch takes what its transfers take).
template <bool E_IN, bool ACT>
__global__ void __launch_bounds__(kThreads, 1)
stage1_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_u,
              const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, stage0 = base + kFwdSlots * kFwdTile, weights = base + 3 * kFwdTile;
    Ring ring = {base, smem_u32(sh.full), kFwdSlots, kFwdTile, p.status, &sh.dead, 0};
    const Sync sync = {sh, p.status, kFwdStages, kFwdSlots};
    const int group = blockIdx.x % kFwdGroups;
    init(sh, p.follows, [&] { sync.load_weights(weights, &tm_w, group * kFwdBlocks, kFwdBlocks); });
    const int first = blockIdx.x / kFwdGroups, step = ranks_of(kFwdGroups, group);
    const int count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    ring.loads = count;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    const Lane ln;
    auto load = [&](int i) {
        if (i >= ring.loads) return;
        if (E_IN) ring.load_linear(i, p.e_in + (size_t)tile(i) * kTileBytes + group * (kFwdBlocks / 8 * kGroupBytes));
        else      ring.load(i, &tm_x, tile(i), group * kFwdBlocks);
    };
    const bool feeder = threadIdx.x == 0;
    if (feeder) {
        for (int i = 0; i < kFwdSlots - 1; ++i)
            if (!p.skips(i)) load(i);
    }
    auto send = [&](int i) {
        store_e(&tm_u, tile(i), stage0 + i % kFwdStages * kFwdTile, group, kFwdBlocks);
    };
    Bias bias;
    if (ACT) bias.load(p.bias, group * kFwdBlocks + ln.warp);
    Weights<4> w;
    sync.take_weights(w, weights + ln.warp * (kM * 128), 0, false);
    if (feeder) {
        sync.wait(sh.w_read, 0, kErrSlotWait);
        load(kFwdSlots - 1);
    }
    // A slot is filled again as soon as its x has been read, one tile before the results have left: 26.1 against 28.0 us forward at
    // 4096 tokens.  With many tiles the launch is bound by DRAM, and reading further ahead costs (block of 32768 tokens 391
    // against 384 us).
    const bool early = count <= 16;
    for (int i = 0; i < count; ++i) {
        const uint32_t x = ring.wait(i), stage = stage0 + i % kFwdStages * kFwdTile;
        uint32_t b[2][2][4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (E_IN) ldm4t(b[v >> 1][v & 1], e_at(x, ln.warp, v >> 1, (v & 1) * 32 + ln.m * 8 + ln.r));
            else      ldm4(b[v >> 1][v & 1], t_at(x, ln.warp, (v >> 1) * 8 + ln.r, (v & 1) * 4 + ln.m));
        }
        if (early) sync.across(i);
        sync.wait_staging(i);
        // a step is 32 rows of 8 tokens; the MMAs of the next one run beside what follows this one's
        float acc[2][2][4];
        auto products = [&](int step) {
#pragma unroll
            for (int k = 0; k < 2; ++k) w.times(2 * (step & 1) + k, b[step >> 1], acc[step & 1][k]);
        };
        products(0);
#pragma unroll
        for (int step = 0; step < 4; ++step) {
            if (step < 3) products(step + 1);
            float (&a)[2][4] = acc[step & 1];
            if (ACT) {
                bias.add(2 * (step & 1), a[0]);
                bias.add(2 * (step & 1) + 1, a[1]);
#pragma unroll
                for (int k = 0; k < 8; k += 2) gelu_fast2(a[k >> 2][k & 3], a[k >> 2][(k & 3) + 1]);
            }
            const int j = (step & 1) * 32 + ln.m * 8 + ln.r;     // row j of this block goes to block j
            stm4(out_at(stage, kFwdBlocks, j, step >> 1, ln.warp), pack_bf16(a[0][0], a[0][1]), pack_bf16(a[0][2], a[0][3]), pack_bf16(a[1][0], a[1][1]),
                 pack_bf16(a[1][2], a[1][3]));
        }
        sync.staged(i);
        if (early && sync.turn(i + 4)) {
            sync.wait_across(i);
            load(i + kFwdSlots);
        }
        sync.pass_on(i, send, [&](int k) {
            if (!early) load(k + kFwdSlots);
        });
    }
    sync.pass_last(count, send);
    sync.leave();
}

// ---------------------------------------------------------------- forward, stage 2: u -> y
// BIAS: y = M x + bias.  Iteration i multiplies tile i + 1 and transposes tile i.
template <bool BIAS>
__global__ void __launch_bounds__(kThreads, 1)
stage2_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_y, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, stage0 = base + kFwdSlots * kFwdTile, weights = base + 3 * kFwdTile;
    Ring ring = {base, smem_u32(sh.full), kFwdSlots, kFwdTile, p.status, &sh.dead, 0};
    const Sync sync = {sh, p.status, kFwdStages, kFwdSlots};
    const int group = blockIdx.x % kFwdGroups;
    init(sh, p.follows, [&] { sync.load_weights(weights, &tm_w, group * kFwdBlocks, kFwdBlocks); });
    const int first = blockIdx.x / kFwdGroups, step = ranks_of(kFwdGroups, group);
    const int count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    ring.loads = count;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    const Lane ln;
    auto load = [&](int i) {
        if (i < ring.loads) ring.load_linear(i, p.e_in + (size_t)tile(i) * kTileBytes + group * (kFwdBlocks / 8 * kGroupBytes));
    };
    const bool feeder = threadIdx.x == 0;
    if (feeder) {
        for (int i = 0; i < kFwdSlots - 1; ++i) load(i);
    }
    auto send = [&](int i) {
        tma_store_3d(&tm_y, stage0 + i % kFwdStages * kFwdTile, group * kFwdBlocks, tile(i) * kTok, 0);
    };
    Weights<4> w;
    sync.take_weights(w, weights + ln.warp * (kM * 128), 0, false);
    if (feeder) {
        sync.wait(sh.w_read, 0, kErrSlotWait);
        load(kFwdSlots - 1);
    }
    Bias bias;
    if (BIAS) bias.load(p.bias, group * kFwdBlocks + ln.warp);
    auto multiply = [&](uint32_t e) {                        // in place: a warp's own block
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t b[2][4], o[8];
#pragma unroll
            for (int v = 0; v < 2; ++v) ldm4t(b[v], e_at(e, ln.warp, h, v * 32 + ln.m * 8 + ln.r));
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                float acc[4];
                w.times(mt, b, acc);
                if (BIAS) bias.add(mt, acc);
                o[2 * mt] = pack_bf16(acc[0], acc[1]);
                o[2 * mt + 1] = pack_bf16(acc[2], acc[3]);
            }
#pragma unroll
            for (int n = 0; n < 2; ++n) stm4(e_at(e, ln.warp, h, n * 32 + ln.m * 8 + ln.r), o[4 * n], o[4 * n + 1], o[4 * n + 2], o[4 * n + 3]);
        }
    };
    if (count > 0) {
        multiply(ring.wait(0));
        sync.across(0);
    }
    for (int i = 0; i < count; ++i) {
        if (i + 1 < count) {
            multiply(ring.wait(i + 1));
            sync.across(i + 1);
        }
        const uint32_t e = ring.slot(i), stage = stage0 + i % kFwdStages * kFwdTile;
        uint32_t v[4][4];
        const int jg = ln.m & 1, h = ln.m >> 1, t = h * 8 + ln.r;
        sync.wait_across(i);
#pragma unroll
        for (int n = 0; n < 4; ++n) ldm4t(v[n], e_at(e, jg * 8 + ln.r, h, ln.warp * 4 + n));
        sync.wait_staging(i);
#pragma unroll
        for (int n = 0; n < 4; ++n) stm4(stage + (ln.warp * 4 + n) * (kTok * 32) + t * 32 + ((jg ^ (t >> 2 & 1)) << 4), v[n]);
        sync.staged(i);
        sync.pass_on(i, send, [&](int k) { load(k + kFwdSlots); });
    }
    sync.pass_last(count, send);
    sync.leave();
}

// ---------------------------------------------------------------- forward on clusters of eight CTAs
// Both stages in one launch: CTA c of a cluster keeps blocks 8 c .. 8 c + 8 of R and of L in registers, a block per warp (warps 0 to
// 7: R, the others: L), and u crosses through distributed shared memory: each warp of stage 1 sends a consumer CTA 256 bytes per
// tile, asynchronously and counted on its barrier, which land as the CTA's 16 KB of an E tile.  So x and y make their one trip and
// u, where the backward call wants it, one more as linear copies.  For small batches, which the two launches of the streams cost
// most (forward of 64 tokens 9.1 -> 6.9 us, block 18.6 -> 12.3 where it was four phases of one launch over units).
// What bounds it, cycles per 16-token tile: MMAs 1030, the exchange 1020 (1860 where the 16-byte pieces of a warp lie 2 KB apart: what
// the order of an E tile is for), y in 16-byte pieces 1200; but a tile takes 2600, most of it the chain of one warp: loads, MMAs,
// transposes, sends and the barriers between.  Taken back, none faster beyond 1500 tokens: half a block of both factors per warp
// (3300 cycles), four more warps that transpose and send (2500), loads of the next tile under the sends (2700).
// Fifteen clusters fit the device (120 of 148 SMs).
//   E_IN    x is E tiles, not token rows          E_OUT  results are E tiles (of the next matrix), not token rows
//   BIAS, GELU                                     SAVE   u is left at p.u_out, as E tiles, for the backward call
constexpr int kCl = 8, kHalfWarps = kWarps / 2;
constexpr int kClX = 3, kClE = 4, kClV = 3, kClY = 3;        // tiles of 16 KB: input slots, exchange slots, w, results
constexpr int kClSmem = (kClX + kClE + 1 + kClV + kClY) * kBwdTile + 1024;
struct ClusterShared {
    uint64_t x_full[kClX], x_read[kClX], e_full[kClE], e_read[kClE], e_free[kClE], across[kClV], staged[8], sent[kClV + kClY], w_full;
    int dead;
};

__device__ __forceinline__ void st_async_16(uint32_t to, uint4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(to), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}

template <bool E_IN, bool E_OUT, bool BIAS, bool GELU, bool SAVE>
__global__ void __launch_bounds__(kThreads, 1)
fwd_cluster_kernel(const __grid_constant__ CUtensorMap tm_R, const __grid_constant__ CUtensorMap tm_L, const __grid_constant__ CUtensorMap tm_x,
                   const __grid_constant__ CUtensorMap tm_y, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ ClusterShared s;
    const uint32_t X0 = (smem_u32(smem_raw) + 1023u) & ~1023u, E0 = X0 + kClX * kBwdTile, U0 = E0 + kClE * kBwdTile, V0 = U0 + kBwdTile;
    constexpr int kOut = E_OUT ? kClV + kClY : kClY;         // result tiles
    const uint32_t Y0 = E_OUT ? V0 : V0 + kClV * kBwdTile;
    const Lane ln;
    const int rank = (int)cluster_ctarank(), lane = threadIdx.x & 31, w = ln.warp & (kHalfWarps - 1), own = rank * kBwdBlocks + w;
    const int first = blockIdx.x / kCl, step = gridDim.x / kCl, count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    // by one lane, or by a warp, whose lanes all learn if one ran out: the warp then does nothing more
    auto wait1 = [&](const uint64_t &bar, int phase, unsigned code) { return mbar_wait(smem_u32(&bar), phase & 1, p.status, &s.dead, code); };
    auto wait = [&](const uint64_t &bar, int phase, unsigned code) { return __all_sync(0xffffffffu, wait1(bar, phase, code)) != 0; };
    // the same on what the other CTAs of the cluster arrive at
    auto wait_cluster = [&](const uint64_t &bar, int phase) {
        return __all_sync(0xffffffffu, mbar_wait<true>(smem_u32(&bar), phase & 1, p.status, &s.dead, kErrPeerWait)) != 0;
    };
    auto turn = [&](int k) { return lane == 0 && (k & (kHalfWarps - 1)) == w; };
    auto arrive = [&](uint64_t &bar) {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar));
    };
    auto load = [&](int i) {
        const uint32_t bar = smem_u32(&s.x_full[i % kClX]), to = X0 + i % kClX * kBwdTile;
        mbar_expect_tx(bar, kBwdTile);
        if (E_IN)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to),
                         "l"(p.e_in + (size_t)tile(i) * kTileBytes + rank * kGroupBytes), "r"(kBwdTile), "r"(bar) : "memory");
        else
            tma_load_3d(to, &tm_x, 0, tile(i) * kTok, rank * kBwdBlocks, bar);
    };
    if (threadIdx.x == 0) {
        for (uint64_t &b : s.x_full) mbar_init(smem_u32(&b), 1);
        for (uint64_t &b : s.x_read) mbar_init(smem_u32(&b), kHalfWarps);
        for (uint64_t &b : s.e_full) mbar_init(smem_u32(&b), 1);
        for (uint64_t &b : s.e_read) mbar_init(smem_u32(&b), kHalfWarps);
        for (uint64_t &b : s.e_free) mbar_init(smem_u32(&b), kCl);
        for (uint64_t &b : s.across) mbar_init(smem_u32(&b), kHalfWarps);
        for (uint64_t &b : s.staged) mbar_init(smem_u32(&b), kHalfWarps);
        for (uint64_t &b : s.sent) mbar_init(smem_u32(&b), 1);
        mbar_init(smem_u32(&s.w_full), 1);
        fence_mbar_init();
        s.dead = 0;
    }
    __syncthreads();
    begin(p.follows, [&] {                                   // into the exchange slots and where the results go
        const uint32_t bar = smem_u32(&s.w_full);
        mbar_expect_tx(bar, 2 * kBwdBlocks * kM * 128);
        for (int b = 0; b < kBwdBlocks; b += 4) {
            tma_load_2d(V0 + b * kM * 128, &tm_R, 0, (rank * kBwdBlocks + b) * kM, bar);
            tma_load_2d(E0 + b * kM * 128, &tm_L, 0, (rank * kBwdBlocks + b) * kM, bar);
        }
    });
    if (threadIdx.x == 0) {
        for (int i = 0; i < kClX && i < count; ++i)
            if (!p.skips(i)) load(i);
        for (int i = 0; i < kClE && i < count; ++i) mbar_expect_tx(smem_u32(&s.e_full[i]), kBwdTile);
    }
    Weights<4> wt;
    bool ok = wait(s.w_full, 0, kErrTmaWait);
    wt.load((ln.warp < kHalfWarps ? V0 : E0) + w * (kM * 128), 0, false);
    cluster_arrive_release();                                // every CTA of the cluster takes the exchange's bytes from here on
    cluster_wait_acquire();

    if (ln.warp < kHalfWarps) {
        // ---- stage 1: u_k = R_k x_k; row j goes to block j, in CTA j / 8
        const uint32_t mine = U0 + w * 2048;
        uint32_t to[2], bar[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = q * 32 + lane;
            to[q] = map_to_cta(e_at(E0, j & 7, 0, own), j >> 3);
            bar[q] = map_to_cta(smem_u32(s.e_full), j >> 3);
        }
        for (int i = 0; ok && i < count; ++i) {
            const uint32_t x = X0 + i % kClX * kBwdTile;
            uint32_t b[2][2][4];
            if (!wait(s.x_full[i % kClX], i / kClX, kErrTmaWait)) break;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (E_IN) ldm4t(b[v >> 1][v & 1], e_at(x, w, v >> 1, (v & 1) * 32 + ln.m * 8 + ln.r));
                else      ldm4(b[v >> 1][v & 1], t_at(x, w, (v >> 1) * 8 + ln.r, (v & 1) * 4 + ln.m));
            }
            arrive(s.x_read[i % kClX]);
            if (i > 0 && turn(i) && i - 1 + kClX < count && wait1(s.x_read[(i - 1) % kClX], (i - 1) / kClX, kErrSlotWait)) load(i - 1 + kClX);
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    float a0[4], a1[4];
                    wt.times(2 * n, b[h], a0);
                    wt.times(2 * n + 1, b[h], a1);
                    stm4(mine + h * 1024 + (n * 32 + ln.m * 8 + ln.r) * 16, pack_bf16(a0[0], a0[1]), pack_bf16(a0[2], a0[3]),
                         pack_bf16(a1[0], a1[1]), pack_bf16(a1[2], a1[3]));
                }
            if (i >= kClE && !wait_cluster(s.e_free[i % kClE], i / kClE - 1)) break;
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint4 v;
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(mine + q * 512 + lane * 16) : "memory");
                st_async_16(to[q & 1] + i % kClE * kBwdTile + (q >> 1) * 128, v, bar[q & 1] + i % kClE * 8);
            }
            __syncwarp();                                    // `mine` has been read
        }
    } else {
        // ---- stage 2: w_j = L_j u_j
        const uint32_t peer_free = map_to_cta(smem_u32(s.e_free), lane & (kCl - 1));
        // Hands tile i's slot back to the eight CTAs, which overwrite it: a release at cluster scope of what this CTA's warps have
        // read, by eight lanes of one warp once they all have.  It costs that warp some 0.5 us, so not by every warp (forward of 1200
        // tokens 16.2 us, 12.9 so), and only where the slot is filled again.
        auto release = [&](int i) {
            if (!wait(s.e_read[i % kClE], i / kClE, kErrMmaWait)) return false;
            if (lane < kCl) mbar_arrive_cluster(peer_free + i % kClE * 8);
            return true;
        };
        Bias bias;
        if (BIAS) bias.load(p.bias, own);
        // put(h, four words of rows 0 .. 31 or 32 .. 63 x 8 tokens, n)
        auto multiply = [&](int i, auto put) {
            const uint32_t e = E0 + i % kClE * kBwdTile;
            if (!wait_cluster(s.e_full[i % kClE], i / kClE)) return false;
            if (threadIdx.x == kHalfWarps * 32 && i + kClE < count) mbar_expect_tx(smem_u32(&s.e_full[i % kClE]), kBwdTile);
            const bool saves = SAVE && turn(i + 4);
            if (saves) {
                fence_proxy_async_smem();
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(p.u_out + (size_t)tile(i) * kTileBytes + rank * kGroupBytes),
                             "r"(e), "r"(kBwdTile) : "memory");
                tma_store_commit();
            }
            __syncwarp();
            uint32_t b[2][2][4];
#pragma unroll
            for (int v = 0; v < 4; ++v) ldm4t(b[v >> 1][v & 1], e_at(e, w, v >> 1, (v & 1) * 32 + ln.m * 8 + ln.r));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t o[8];
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    float acc[4];
                    wt.times(mt, b[h], acc);
                    if (BIAS) bias.add(mt, acc);
                    if (GELU) {
                        gelu_fast2(acc[0], acc[1]);
                        gelu_fast2(acc[2], acc[3]);
                    }
                    o[2 * mt] = pack_bf16(acc[0], acc[1]);
                    o[2 * mt + 1] = pack_bf16(acc[2], acc[3]);
                }
                if (!put(h, o)) return false;
            }
            // (after the products: the tile is in registers)  By turns, a tile later: the others have read it, and so has its copy.
            arrive(s.e_read[i % kClE]);
            if (i > 0 && w == ((i + 3) & (kHalfWarps - 1))) {
                if (SAVE && lane == 0) tma_store_wait_read<0>();
                __syncwarp();
                if (i - 1 + kClE < count && !release(i - 1)) return false;
            }
            return true;
        };
        auto send = [&](int i) {
            const uint32_t from = Y0 + i % kOut * kBwdTile;
            if (E_OUT)                                       // (one tensor copy instead: block of 512 tokens 20.1 against 19.4 us)
#pragma unroll
                for (int g = 0; g < kM / 8; ++g)
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(p.e_out + (size_t)tile(i) * kTileBytes + g * kGroupBytes + rank * (kBwdBlocks * kRowBytes)),
                                 "r"(from + g * (kBwdBlocks * kRowBytes)), "r"(kBwdBlocks * kRowBytes) : "memory");
            else
                tma_store_3d(&tm_y, from, rank * kBwdBlocks, tile(i) * kTok, 0);
            tma_store_commit();
        };
        // results of tile i are in their tile; the ones before leave, by turns
        auto pass_on = [&](int i) {
            fence_proxy_async_smem();
            arrive(s.staged[i & 7]);
            if (i >= 2 && turn(i - 2)) {
                tma_store_wait_read<0>();
                mbar_arrive(smem_u32(&s.sent[(i - 2) % kOut]));
            }
            if (i >= 1 && turn(i - 1) && wait1(s.staged[(i - 1) & 7], (i - 1) >> 3, kErrMmaWait)) send(i - 1);
            __syncwarp();
        };
        auto wait_sent = [&](int i) { return i < kOut || wait(s.sent[i % kOut], i / kOut - 1, kErrSlotWait); };
        int i = 0;
        if (E_OUT) {
            for (; ok && i < count; ++i) {
                const uint32_t out = Y0 + i % kOut * kBwdTile;
                if (!multiply(i, [&](int h, const uint32_t (&o)[8]) {
                        if (h == 0 && !wait_sent(i)) return false;
#pragma unroll
                        for (int n = 0; n < 2; ++n) stm4(out_at(out, kBwdBlocks, n * 32 + ln.m * 8 + ln.r, h, w), o[4 * n], o[4 * n + 1], o[4 * n + 2], o[4 * n + 3]);
                        return true;
                    }))
                    break;
                pass_on(i);
            }
        } else {
            auto ahead = [&](int k) {                        // w, as an E tile: transposed below
                const uint32_t V = V0 + k % kClV * kBwdTile;
                if (!multiply(k, [&](int h, const uint32_t (&o)[8]) {
                        if (h == 0 && k >= kClV && !wait(s.staged[(k - kClV) & 7], (k - kClV) >> 3, kErrMmaWait)) return false;
#pragma unroll
                        for (int n = 0; n < 2; ++n) stm4(e_at(V, w, h, n * 32 + ln.m * 8 + ln.r), o[4 * n], o[4 * n + 1], o[4 * n + 2], o[4 * n + 3]);
                        return true;
                    }))
                    return false;
                arrive(s.across[k % kClV]);
                return true;
            };
            ok = ok && (count == 0 || ahead(0));
            for (; ok && i < count; ++i) {
                if (i + 1 < count && !ahead(i + 1)) break;
                const uint32_t V = V0 + i % kClV * kBwdTile, out = Y0 + i % kOut * kBwdTile;
                if (!wait(s.across[i % kClV], i / kClV, kErrMmaWait)) break;
                uint32_t v[4][4];
                const int h = ln.m & 1, lo = ln.m >> 1;
#pragma unroll
                for (int n = 0; n < 4; ++n) ldm4t(v[n], e_at(V, ln.r, h, w * 8 + n * 2 + lo));
                if (!wait_sent(i)) break;
#pragma unroll
                for (int n = 0; n < 4; ++n) stm4(out + (w * 8 + n * 2 + lo) * (kTok * 16) + (h * 8 + ln.r) * 16, v[n]);
                pass_on(i);
            }
        }
        if (i == count && count > 0 && turn(count - 1) && wait1(s.staged[(count - 1) & 7], (count - 1) >> 3, kErrMmaWait)) send(count - 1);
        tma_store_wait_all<0>();
    }
    let_copies_land(&s.dead);
    __syncthreads();
    cluster_arrive_release();                                // nobody leaves while others may still write here
    cluster_wait_acquire();
}

// ---------------------------------------------------------------- backward
// sums of rows half * 32 .. + 32 and all 64 columns of a warp's block: A = rows of an E block, B = rows of an E block or
// columns of a T tile, both by token
struct Sums {
    float v[2][8][4];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i >> 5][i >> 2 & 7][i & 3] = 0.0f;
    }
    template <bool BT> __device__ __forceinline__ void add(uint32_t A, uint32_t B, int blk, int half)
    {
        const Lane ln;
        uint32_t a[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) ldm4(a[mt], e_at(A, blk, ln.m >> 1, half * 32 + mt * 16 + (ln.m & 1) * 8 + ln.r));
#pragma unroll
        for (int np = 0; np < 4; ++np) {
            uint32_t b[4];
            const int col = np * 2 + (ln.m >> 1), h = ln.m & 1;
            if (BT) ldm4t(b, t_at(B, blk, h * 8 + ln.r, col));
            else    ldm4(b, e_at(B, blk, h, col * 8 + ln.r));
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                mma(v[mt][2 * np], a[mt], b[0], b[1]);
                mma(v[mt][2 * np + 1], a[mt], b[2], b[3]);
            }
        }
    }
    __device__ __forceinline__ void store(float *block, int half) const
    {
        const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 *to = reinterpret_cast<float2 *>(block + (half * 32 + mt * 16 + g + 8 * h) * kM + nt * 8 + 2 * q);
                    *to = make_float2(v[mt][nt][2 * h], v[mt][nt][2 * h + 1]);
                }
    }
};

// dy -> z, du (E tiles) and, with DW, dL.  Iteration i: z(i + 1), du(i), sums of tile i.
template <bool DW>
__global__ void __launch_bounds__(kThreads, 1)
bwd_du_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_dy, const __grid_constant__ CUtensorMap tm_du,
              const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, V0 = base + kDuSlots * kBwdTile, stage0 = V0 + 3 * kBwdTile;
    const uint32_t weights = base + 10 * kBwdTile;
    Ring ring = {base, smem_u32(sh.full), kDuSlots, kBwdTile, p.status, &sh.dead, 0};
    const Sync sync = {sh, p.status, kDuStages, 3};
    const int group = blockIdx.x % kBwdGroups;
    init(sh, p.follows, [&] { sync.load_weights(weights, &tm_w, group * kBwdBlocks, kBwdBlocks); });
    const int first = blockIdx.x / kBwdGroups, step = ranks_of(kBwdGroups, group);
    const int count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    ring.loads = (DW ? 2 : 1) * count;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    constexpr int kItems = DW ? 2 : 1;                       // per tile: dy, u
    const Lane ln;
    auto load = [&](int from, int to) {
        for (int i = from; i <= to && i < ring.loads; ++i) {
            const int t = tile(i / kItems);
            if (DW && (i & 1)) ring.load_linear(i, p.u + (size_t)t * kTileBytes + group * kGroupBytes);
            else               ring.load(i, &tm_dy, t, 0, group * kBwdBlocks);
        }
    };
    const bool feeder = threadIdx.x == 0;
    if (feeder) {
        for (int i = 0; i < kDuSlots; ++i)
            if (!p.skips(i)) load(i, i);
    }
    auto send = [&](int i) {
        store_e(&tm_du, tile(i), stage0 + i % kDuStages * kBwdTile, group, kBwdBlocks);
    };
    auto refill = [&](int i) {                               // dy(i + 1) and u(i) have been read
        load(i == 0 ? kDuSlots : kItems * i + 1 + kDuSlots, kItems * (i + 1) + kDuSlots);
    };
    const int blk = ln.warp >> 1, half = ln.warp & 1;
    Weights<2> w;
    sync.take_weights(w, weights + blk * (kM * 128), half * 32, true);
    Sums sums;
    if (DW) sums.clear();
    // [l][token][8 columns j] -> E blocks [j][l]
    auto transpose = [&](uint32_t y, uint32_t V) {
        uint32_t v[2][4];
        const int h = ln.m & 1, lo = ln.m >> 1;
#pragma unroll
        for (int n = 0; n < 2; ++n) ldm4t(v[n], y + (ln.warp * 4 + n * 2 + lo) * (kTok * 16) + (h * 8 + ln.r) * 16);
#pragma unroll
        for (int n = 0; n < 2; ++n) stm4(e_at(V, ln.r, h, ln.warp * 4 + n * 2 + lo), v[n]);
    };
    if (count > 0) {
        sync.wait(sh.w_read, 0, kErrSlotWait);               // V(2) lies where the weights were
        transpose(ring.wait(0), V0);
        sync.across(0);
    }
    for (int i = 0; i < count; ++i) {
        const uint32_t V = V0 + i % 3 * kBwdTile, stage = stage0 + i % kDuStages * kBwdTile;
        if (i + 1 < count) {
            const uint32_t y = ring.wait(kItems * (i + 1));
            if (i > 1) sync.wait_staged(i - 2);              // every warp is done with V(i - 2)
            transpose(y, V0 + (i + 1) % 3 * kBwdTile);
            sync.across(i + 1);
        }
        sync.wait_across(i);
        uint32_t b[2][2][4];
#pragma unroll
        for (int v = 0; v < 4; ++v) ldm4t(b[v >> 1][v & 1], e_at(V, blk, v >> 1, (v & 1) * 32 + ln.m * 8 + ln.r));
        sync.wait_staging(i);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float a0[4], a1[4];
            w.times(0, b[h], a0);
            w.times(1, b[h], a1);
            const int k = half * 32 + ln.m * 8 + ln.r;       // row k of this block goes to block k
            stm4(out_at(stage, kBwdBlocks, k, h, blk), pack_bf16(a0[0], a0[1]), pack_bf16(a0[2], a0[3]),
                 pack_bf16(a1[0], a1[1]), pack_bf16(a1[2], a1[3]));
        }
        if (DW) sums.add<false>(V, ring.wait(2 * i + 1), blk, half);
        sync.staged(i);
        sync.pass_on(i, send, refill);
    }
    sync.pass_last(count, send);
    if (DW && count > 0)
        sums.store(p.parts + (size_t)first * kGradElems + (size_t)(group * kBwdBlocks + blk) * kM * kM, half);
    sync.leave();
}

// du -> dx (DX) and dR (DW)
template <bool DX, bool DW>
__global__ void __launch_bounds__(kThreads, 1)
bwd_dx_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dx,
              const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, stage0 = base + kDxSlots * kBwdTile;
    Ring ring = {base, smem_u32(sh.full), kDxSlots, kBwdTile, p.status, &sh.dead, 0};
    const Sync sync = {sh, p.status, DX ? kDxStages : kMaxStages, 1};   // without staging, warps are up to five tiles apart
    const int group = blockIdx.x % kBwdGroups;
    init(sh, p.follows, [&] {
        if (DX) sync.load_weights(stage0, &tm_w, group * kBwdBlocks, kBwdBlocks);
    });
    const int first = blockIdx.x / kBwdGroups, step = ranks_of(kBwdGroups, group);
    const int count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    ring.loads = (DW ? 2 : 1) * count;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    constexpr int kItems = DW ? 2 : 1;                       // per tile: du, x
    const Lane ln;
    auto load = [&](int from, int to) {
        for (int i = from; i <= to && i < ring.loads; ++i) {
            const int t = tile(i / kItems);
            if (DW && (i & 1)) ring.load(i, &tm_x, t, group * kBwdBlocks);
            else               ring.load_linear(i, p.e_in + (size_t)t * kTileBytes + group * kGroupBytes);
        }
    };
    const bool feeder = threadIdx.x == 0;
    if (feeder) load(0, kDxSlots - 1);
    auto send = [&](int i) {
        if (DX) tma_store_3d(&tm_dx, stage0 + i % kDxStages * kBwdTile, 0, tile(i) * kTok, group * kBwdBlocks);
    };
    const int blk = ln.warp >> 1, half = ln.warp & 1;
    Weights<2> w;
    if (DX) sync.take_weights(w, stage0 + blk * (kM * 128), half * 32, true);
    Sums sums;
    if (DW) sums.clear();
    for (int i = 0; i < count; ++i) {
        const uint32_t du = ring.wait(kItems * i), stage = stage0 + i % kDxStages * kBwdTile;
        if (DX) {
            uint32_t b[2][2][4];
#pragma unroll
            for (int v = 0; v < 4; ++v) ldm4t(b[v >> 1][v & 1], e_at(du, blk, v >> 1, (v & 1) * 32 + ln.m * 8 + ln.r));
            sync.wait_staging(i);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float a0[4], a1[4];
                w.times(0, b[h], a0);
                w.times(1, b[h], a1);
                const uint32_t o[4] = {pack_bf16(a0[0], a0[1]), pack_bf16(a0[2], a0[3]), pack_bf16(a1[0], a1[1]), pack_bf16(a1[2], a1[3])};
                stm4t(t_at(stage, blk, h * 8 + ln.r, half * 4 + ln.m), o);
            }
        }
        if (DW) sums.add<true>(du, ring.wait(2 * i + 1), blk, half);
        sync.staged(i);
        sync.pass_on(i, send, [&](int k) { load(kItems * k + kDxSlots, kItems * (k + 1) - 1 + kDxSlots); });
    }
    sync.pass_last(count, send);
    if (DW && count > 0)
        sums.store(p.parts + (size_t)first * kGradElems + (size_t)(group * kBwdBlocks + blk) * kM * kM, half);
    sync.leave();
}

// grads = (accumulate ? grads : 0) + the parts of every rank, in order; 64 groups of 4 elements and 4 ranges of ranks per CTA
// (all ranks by one thread, 19 loads in flight and a quarter of the CTAs: 20 us against 12)
__global__ void __launch_bounds__(256)
add_parts_m64_kernel(const float *__restrict__ parts_l, const float *__restrict__ parts_r, float *__restrict__ dL, float *__restrict__ dR,
                     int grid, int accumulate)
{
    __shared__ float4 red[4][64];
    constexpr int kPer = 64 * 4, kCtas = (int)(kGradElems / kPer);
    const int kind = blockIdx.x / kCtas, at = blockIdx.x % kCtas * kPer + (threadIdx.x & 63) * 4, range = threadIdx.x >> 6;
    const int group = at / (kBwdBlocks * kM * kM), n = (grid - group + kBwdGroups - 1) / kBwdGroups, per = (n + 3) / 4;
    const float *src = (kind == 0 ? parts_l : parts_r) + at;
    float *dst = (kind == 0 ? dL : dR) + at;
    float4 s = make_float4(0, 0, 0, 0);
    depend_wait();
    // What follows takes the SMs over as they empty (forward + backward of 500 tokens 36 -> 34 us, 2000 60.1 -> 56.7, 8192 142 -> 137;
    // the feed-forward block's 500 tokens 92 -> 89, 3000 210.5 -> 208.5, 6000 333 -> 334.5, 8192 426 -> 429); with fewer parts to add
    // its blocks are only in the way (64 tokens 23.5 -> 23.8).
    if (n >= 8) depend_launch();
#pragma unroll 5
    for (int i = range * per; i < (range + 1) * per && i < n; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(src + (size_t)i * kGradElems);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    red[range][threadIdx.x & 63] = s;
    __syncthreads();
    if (range == 0) {
        if (accumulate) {
            const float4 o = *reinterpret_cast<const float4 *>(dst);
            s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
        }
#pragma unroll
        for (int i = 1; i < 4; ++i) {
            const float4 v = red[i][threadIdx.x];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4 *>(dst) = s;
    }
}

// ---------------------------------------------------------------- complex factors
// One stage of y = M x (FIRST != PERM) or y = M^H x (FIRST == PERM) with planar complex tensors: FIRST reads token rows and
// leaves E tiles, the other way round otherwise; PERM: the token rows are the permuted side (the forward's output, the
// adjoint's input).  A CTA keeps both planes of 8 blocks, so the four real products of a stage add up in the accumulators and
// the intermediate is rounded once; as four real calls on the stacked planes and a combining pass this took twice the MMAs and
// 5 x the memory traffic (2048 tokens, M^H (M x): 293 us, now 87; 64 tokens 72, now 21.6).
template <bool FIRST, bool PERM>
__global__ void __launch_bounds__(kThreads, 1)
cplx_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_e, const __grid_constant__ CUtensorMap tm_re,
            const __grid_constant__ CUtensorMap tm_im, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    constexpr bool kAdjoint = FIRST == PERM;
    // a pair of 16 KB tiles (re, im) per token tile: input slots, transposed tiles, staging; the weights come first, into the last 128 KB
    constexpr int kPair = 2 * kBwdTile, kTiles = PERM ? 3 : 4, kStages = PERM ? 2 : 3;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, V0 = base + kTiles * kPair, stage0 = V0 + (PERM ? 2 * kPair : 0);
    const uint32_t weights = base + 3 * kPair;
    Ring ring = {base, smem_u32(sh.full), 2 * kTiles, kBwdTile, p.status, &sh.dead, 0};
    const Sync sync = {sh, p.status, kStages, 2};
    const int group = blockIdx.x % kBwdGroups;
    init(sh, p.follows, [&] { sync.load_weights(weights, &tm_w, group * kBwdBlocks, kBwdBlocks, 2); });
    const int first = blockIdx.x / kBwdGroups, step = ranks_of(kBwdGroups, group);
    const int count = first < p.tiles ? (p.tiles - first + step - 1) / step : 0;
    ring.loads = 2 * count;
    auto tile = [&](int i) { return p.last != 0 ? p.last - first - i * step : first + i * step; };
    const Lane ln;
    const int blk = ln.warp >> 1, half = ln.warp & 1;
    auto load = [&](int i) {
        if (2 * i >= ring.loads) return;
        const int t = tile(i);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (!FIRST)    ring.load_linear(2 * i + c, p.e_in + (size_t)(c * p.tiles + t) * kTileBytes + group * kGroupBytes);
            else if (PERM) ring.load(2 * i + c, c ? &tm_im : &tm_re, t, 0, group * kBwdBlocks);
            else           ring.load(2 * i + c, c ? &tm_im : &tm_re, t, group * kBwdBlocks);
        }
    };
    const bool feeder = threadIdx.x == 0;
    if (feeder) {
        for (int i = 0; i < 3; ++i)
            if (!p.skips(i)) load(i);
    }
    Weights<2> wr, wi;
    sync.wait(sh.w_full, 0, kErrTmaWait);
    wr.load(weights + blk * (kM * 128), half * 32, kAdjoint);
    wi.load(weights + (kBwdBlocks + blk) * (kM * 128), half * 32, kAdjoint);
    sync.arrive(sh.w_read);
    if (kAdjoint)
#pragma unroll
        for (int k = 0; k < 32; ++k) wi.a[k >> 4][k >> 2 & 3][k & 3] ^= 0x80008000u;
    sync.wait(sh.w_read, 0, kErrSlotWait);
    if (feeder && !PERM) load(3);

    // put(h, plane, four words of 32 outputs x 8 tokens) of this warp's rows
    auto product = [&](uint32_t re, uint32_t im, auto put) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t x[2][2][4];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    if (FIRST && !PERM) ldm4(x[c][v], t_at(c ? im : re, blk, h * 8 + ln.r, v * 4 + ln.m));
                    else                ldm4t(x[c][v], e_at(c ? im : re, blk, h, v * 32 + ln.m * 8 + ln.r));
                }
            float a[2][2][4];
#pragma unroll
            for (int k = 0; k < 16; ++k) a[k >> 3][k >> 2 & 1][k & 3] = 0.0f;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const uint32_t r0 = x[0][ks >> 1][(ks & 1) * 2], r1 = x[0][ks >> 1][(ks & 1) * 2 + 1];
                const uint32_t i0 = x[1][ks >> 1][(ks & 1) * 2], i1 = x[1][ks >> 1][(ks & 1) * 2 + 1];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    mma(a[0][mt], wr.a[mt][ks], r0, r1);
                    mma(a[1][mt], wr.a[mt][ks], i0, i1);
                    mma(a[0][mt], wi.a[mt][ks], i0 ^ 0x80008000u, i1 ^ 0x80008000u);
                    mma(a[1][mt], wi.a[mt][ks], r0, r1);
                }
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t o[4] = {pack_bf16(a[c][0][0], a[c][0][1]), pack_bf16(a[c][0][2], a[c][0][3]), pack_bf16(a[c][1][0], a[c][1][1]),
                                       pack_bf16(a[c][1][2], a[c][1][3])};
                put(h, c, o);
            }
        }
    };
    // what PERM does one tile ahead: token rows -> V, or E tile -> product -> V
    auto ahead = [&](int i) {
        const uint32_t re = ring.wait(2 * i), im = ring.wait(2 * i + 1), V = V0 + (i & 1) * kPair;
        if (i > 1) sync.wait_staged(i - 2);                  // every warp is done with V(i - 2)
        if constexpr (FIRST) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t v[2][4];
                const int h = ln.m & 1, lo = ln.m >> 1;
#pragma unroll
                for (int n = 0; n < 2; ++n) ldm4t(v[n], (c ? im : re) + (ln.warp * 4 + n * 2 + lo) * (kTok * 16) + (h * 8 + ln.r) * 16);
#pragma unroll
                for (int n = 0; n < 2; ++n) stm4(e_at(V + c * kBwdTile, ln.r, h, ln.warp * 4 + n * 2 + lo), v[n]);
            }
        } else {
            product(re, im, [&](int h, int c, const uint32_t (&o)[4]) { stm4(e_at(V + c * kBwdTile, blk, h, half * 32 + ln.m * 8 + ln.r), o); });
        }
        sync.across(i);
    };
    auto send = [&](int k) {
        const int t = tile(k);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const uint32_t from = stage0 + k % kStages * kPair + c * kBwdTile;
            if (FIRST)     store_e(&tm_e, c * p.tiles + t, from, group, kBwdBlocks);
            else if (PERM) tma_store_3d(c ? &tm_im : &tm_re, from, group * kBwdBlocks, t * kTok, 0);
            else           tma_store_3d(c ? &tm_im : &tm_re, from, 0, t * kTok, group * kBwdBlocks);
        }
    };
    if (PERM && count > 0) ahead(0);
    for (int i = 0; i < count; ++i) {
        const uint32_t stage = stage0 + i % kStages * kPair;
        uint32_t re = V0 + (i & 1) * kPair, im = re + kBwdTile;
        if constexpr (PERM) {
            if (i + 1 < count) ahead(i + 1);
            sync.wait_across(i);
        } else {
            re = ring.wait(2 * i);
            im = ring.wait(2 * i + 1);
        }
        sync.wait_staging(i);
        if constexpr (!FIRST && PERM) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t v[2][4];
                const int h = ln.m & 1, lo = ln.m >> 1;
#pragma unroll
                for (int n = 0; n < 2; ++n) ldm4t(v[n], e_at(c ? im : re, ln.r, h, ln.warp * 4 + n * 2 + lo));
#pragma unroll
                for (int n = 0; n < 2; ++n) stm4(stage + c * kBwdTile + (ln.warp * 4 + n * 2 + lo) * (kTok * 16) + (h * 8 + ln.r) * 16, v[n]);
            }
        } else {
            product(re, im, [&](int h, int c, const uint32_t (&o)[4]) {
                const int k = half * 32 + ln.m * 8 + ln.r;
                if (FIRST) stm4(out_at(stage + c * kBwdTile, kBwdBlocks, k, h, blk), o);
                else       stm4t(t_at(stage + c * kBwdTile, blk, h * 8 + ln.r, half * 4 + ln.m), o);
            });
        }
        sync.staged(i);
        sync.pass_on(i, send, [&](int k) {
            if (PERM && k == 0) load(3);
            load(k + 4);                                     // PERM: of three slots, tile k + 1's
        });
    }
    sync.pass_last(count, send);
    sync.leave();
}

// ---------------------------------------------------------------- host
// [tokens][4096] as boxes of 64 columns: a copy of 64 columns x 16 tokens x `blocks` boxes is a T tile
int map_t(CUtensorMap *m, const void *p, int64_t tokens, int blocks)
{
    const uint64_t dims[3] = {kM, (uint64_t)tokens, kM}, strides[2] = {kN * 2, kM * 2};
    const uint32_t box[3] = {kM, kTok, (uint32_t)blocks};
    return encode_tmap_nd(m, p, 2, 3, dims, strides, box, 128);
}
// the same tensor as [l][t][j]: `columns` neighbouring j of every l
int map_y(CUtensorMap *m, const void *p, int64_t tokens, int columns)
{
    const uint64_t dims[3] = {kM, (uint64_t)tokens, kM}, strides[2] = {kN * 2, kM * 2};
    const uint32_t box[3] = {(uint32_t)columns, kTok, kM};
    return encode_tmap_nd(m, p, 2, 3, dims, strides, box, columns == 16 ? 32 : 0);
}
// E tiles as (tile, 8 consumers) x 8 producers x 2 KB: the pieces of `blocks` producers in all groups of a tile.  (As eight linear
// copies of a thread per tile the complex multiply of 8192 tokens took 306 us, as one tensor
// copy 288; as 256-byte pieces, in the order [consumer][half][producer], 295.)
int map_e(CUtensorMap *m, const void *p, int tiles, int blocks)
{
    constexpr uint32_t kPiece = 8 * kRowBytes;
    const uint64_t dims[3] = {kPiece / 8, 8, (uint64_t)tiles * (kM / 8)}, strides[2] = {kPiece, kGroupBytes};
    const uint32_t box[3] = {kPiece / 8, (uint32_t)blocks / 8, kM / 8};
    return encode_tmap_nd(m, p, 8, 3, dims, strides, box);
}
// blocks as rows of 64 columns, four blocks a copy
int map_w(CUtensorMap *m, const void *W, int planes = 1) { return encode_tmap_2d(m, W, planes * kN, kM, kM * 2, 4 * kM, kM, 128); }

int64_t tiles_of(int64_t tokens) { return (tokens + kTok - 1) / kTok; }
size_t max_ranks(int64_t tokens) { return (size_t)(tiles_of(tokens) < kMaxRanks ? tiles_of(tokens) : kMaxRanks); }
size_t e_bytes(int64_t tokens) { return (size_t)tiles_of(tokens) * kTileBytes; }

int grid_of(int groups, int sms, int64_t tokens)
{
    const int64_t all = tiles_of(tokens) * groups;
    return (int)(all < sms ? all : sms);
}

// x: token rows or E tiles; u: E tiles
template <bool E_IN, bool ACT>
int stage1(const void *x, const void *W, const void *bias, void *u, int64_t tokens, int follows, bool backwards, int sms, unsigned *status, cudaStream_t s)
{
    CUtensorMap tm_w, tm_x = {}, tm_u;
    MONARCH_TRY(map_w(&tm_w, W));
    MONARCH_TRY(map_e(&tm_u, u, (int)tiles_of(tokens), kFwdBlocks));
    if (!E_IN) MONARCH_TRY(map_t(&tm_x, x, tokens, kFwdBlocks));
    Params p = {};
    p.skip = follows ? -1 : take_skipped_tile();
    p.follows = follows;
    p.status = status;
    p.bias = (const __nv_bfloat16 *)bias;
    p.e_in = (const char *)x;
    p.tiles = (int)tiles_of(tokens);
    p.last = backwards ? p.tiles - 1 : 0;
    return launch_serialized(stage1_kernel<E_IN, ACT>, grid_of(kFwdGroups, sms, tokens), kThreads, kFwdSmem, s, tm_w, tm_x, tm_u, p);
}
int stage2(const void *u, const void *W, const void *bias, void *y, int64_t tokens, int sms, unsigned *status, cudaStream_t s)
{
    CUtensorMap tm_w, tm_y;
    MONARCH_TRY(map_w(&tm_w, W));
    MONARCH_TRY(map_y(&tm_y, y, tokens, kFwdBlocks));
    Params p = {};
    p.skip = -1;
    p.follows = 1;
    p.status = status;
    p.bias = (const __nv_bfloat16 *)bias;
    p.e_in = (const char *)u;
    p.tiles = (int)tiles_of(tokens);
    p.last = p.tiles - 1;
    return launch_serialized(bias != nullptr ? stage2_kernel<true> : stage2_kernel<false>, grid_of(kFwdGroups, sms, tokens), kThreads, kFwdSmem, s,
                             tm_w, tm_y, p);
}

// Launch attributes of a cluster kernel, and how many clusters fit the device at once (0: none do)
struct ClusterLaunch {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg;
    explicit ClusterLaunch(cudaStream_t s) : cfg()
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kCl;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.blockDim = dim3(kThreads);
        cfg.gridDim = dim3(kCl);
        cfg.dynamicSmemBytes = kClSmem;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};
template <bool E_IN, bool E_OUT, bool BIAS, bool GELU, bool SAVE> int clusters()
{
    static PerDeviceCache fit;
    auto kern = fwd_cluster_kernel<E_IN, E_OUT, BIAS, GELU, SAVE>;
    int n = fit.get();
    if (n < 0) {
        const ClusterLaunch launch(nullptr);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kClSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &launch.cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        fit.set(n);
    }
    return n;
}

// One multiply on clusters; x, y: token rows or E tiles
template <bool E_IN, bool E_OUT, bool BIAS, bool GELU, bool SAVE>
int fwd_on_clusters(const void *x, const void *L, const void *R, const void *bias, void *y, void *u, int64_t tokens, bool follows, unsigned *status,
                    cudaStream_t s)
{
    const int64_t fit = clusters<E_IN, E_OUT, BIAS, GELU, SAVE>();
    if (fit <= 0) return MONARCH_ERR_UNSUPPORTED;
    ClusterLaunch launch(s);
    launch.cfg.numAttrs = 2;
    launch.cfg.gridDim = dim3((unsigned)(kCl * (tiles_of(tokens) < fit ? tiles_of(tokens) : fit)));
    CUtensorMap tm_R, tm_L, tm_x = {}, tm_y = {};
    MONARCH_TRY(map_w(&tm_R, R));
    MONARCH_TRY(map_w(&tm_L, L));
    if (!E_IN) MONARCH_TRY(map_t(&tm_x, x, tokens, kBwdBlocks));
    if (!E_OUT) MONARCH_TRY(map_y(&tm_y, y, tokens, kBwdBlocks));
    Params p = {};
    p.skip = take_skipped_tile();
    p.status = status;
    p.bias = (const __nv_bfloat16 *)bias;
    p.e_in = (const char *)x;
    p.e_out = (char *)y;
    p.u_out = (char *)u;
    p.tiles = (int)tiles_of(tokens);
    p.follows = follows;
    p.last = follows ? p.tiles - 1 : 0;
    MONARCH_CUDA_TRY(cudaLaunchKernelEx(&launch.cfg, fwd_cluster_kernel<E_IN, E_OUT, BIAS, GELU, SAVE>, tm_R, tm_L, tm_x, tm_y, p));
    note_launch();
    return MONARCH_OK;
}

}  // namespace
}  // namespace tc

// Where the forward runs on clusters.  They take 5.6 us and 1.45 for every round of tiles, of which there are as many as clusters
// fit (15); the streams, in which a tile takes four CTAs, 8 us as long as each CTA has one.  So: one round, or more tiles than
// the streams' CTAs, up to five rounds (us, clusters / streams: 240 tokens 6.9 / 8.3, 300 8.6 / 8.4, 600 9.8 / 11.7, 960
// 11.6 / 13.1, 1500 16.2 / 15.8).  Under the feed-forward backward, whose next launch reads y, one round (1000 tokens 122.8 / 121.7).
static bool fwd_prefers_clusters(int64_t tokens, bool bias, int sms)
{
    const int64_t tiles = tc::tiles_of(tokens), fit = bias ? tc::clusters<false, false, true, false, true>() : tc::clusters<false, false, false, false, true>();
    return fit > 0 && (tiles <= fit || (!bias && tiles * tc::kFwdGroups > sms && tiles <= 5 * fit));
}
// The feed-forward block, whose streams are four launches, up to ten rounds (16 tokens 11.5 / 17.4, 1000 24.9 / 28.9, 2400 40.5 /
// 42.5, 2700 45.5 / 44.3)
static bool mlp_prefers_clusters(int64_t tokens)
{
    const int64_t fit = tc::clusters<false, true, true, true, false>(), last = tc::clusters<true, false, true, false, false>();
    return fit > 0 && last > 0 && tc::tiles_of(tokens) <= 10 * fit;
}

// y = M x + bias (bias null: y = M x); u: E tiles of all tokens, kept for the backward call
static int stream_fwd(const void *x, const void *L, const void *R, const void *bias, void *y, void *u, int64_t tokens, unsigned *status, cudaStream_t s)
{
    using namespace tc;
    if (tokens == 0) return MONARCH_OK;
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    if (fwd_prefers_clusters(tokens, bias != nullptr, sms))
        return bias != nullptr ? fwd_on_clusters<false, false, true, false, true>(x, L, R, bias, y, u, tokens, false, status, s)
                               : fwd_on_clusters<false, false, false, false, true>(x, L, R, nullptr, y, u, tokens, false, status, s);
    MONARCH_TRY((stage1<false, false>(x, R, nullptr, u, tokens, 0, false, sms, status, s)));
    return stage2(u, L, bias, y, tokens, sms, status, s);
}

// dx null: gradients only; dL null: dx only.  u: what the forward call left (u_saved), or scratch for E tiles of all tokens;
// du: scratch of the same size; parts: two gradients of max_ranks(tokens)
static int stream_bwd(const void *x, const void *dy, const void *L, const void *R, const void *u, bool u_saved, void *dx, float *dL, float *dR,
                      int accumulate, void *du, void *parts, int64_t tokens, unsigned *status, cudaStream_t s)
{
    using namespace tc;
    if (tokens == 0) {
        if (dL != nullptr && !accumulate) {
            MONARCH_CUDA_TRY(cudaMemsetAsync(dL, 0, kGradElems * sizeof(float), s));
            MONARCH_CUDA_TRY(cudaMemsetAsync(dR, 0, kGradElems * sizeof(float), s));
        }
        return MONARCH_OK;
    }
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    if (sms > kMaxRanks * kBwdGroups) sms = kMaxRanks * kBwdGroups;
    float *parts_l = (float *)parts, *parts_r = parts_l + max_ranks(tokens) * kGradElems;
    const int grid = grid_of(kBwdGroups, sms, tokens), tiles = (int)tiles_of(tokens);
    if (dL != nullptr && !u_saved) MONARCH_TRY((stage1<false, false>(x, R, nullptr, (void *)u, tokens, 0, false, sms, status, s)));
    CUtensorMap tm_L, tm_R, tm_dy, tm_du, tm_x, tm_dx;
    MONARCH_TRY(map_w(&tm_L, L));
    MONARCH_TRY(map_w(&tm_R, R));
    MONARCH_TRY(map_y(&tm_dy, dy, tokens, kBwdBlocks));
    MONARCH_TRY(map_e(&tm_du, du, tiles, kBwdBlocks));
    MONARCH_TRY(map_t(&tm_x, dL != nullptr ? x : dy, tokens, kBwdBlocks));
    MONARCH_TRY(map_t(&tm_dx, dx != nullptr ? dx : dy, tokens, kBwdBlocks));
    Params p = {};
    p.skip = take_skipped_tile();
    p.status = status;
    p.u = (const char *)u;
    p.parts = parts_l;
    p.tiles = tiles;
    MONARCH_TRY(launch_serialized(dL != nullptr ? bwd_du_kernel<true> : bwd_du_kernel<false>, grid, kThreads, kBwdSmem, s, tm_L, tm_dy, tm_du, p));
    p.skip = -1;
    p.follows = 1;
    p.e_in = (const char *)du;
    p.parts = parts_r;
    p.last = tiles - 1;
    auto last = dx == nullptr ? bwd_dx_kernel<false, true> : dL == nullptr ? bwd_dx_kernel<true, false> : bwd_dx_kernel<true, true>;
    MONARCH_TRY(launch_serialized(last, grid, kThreads, kBwdSmem, s, tm_R, tm_x, tm_dx, p));
    if (dL == nullptr) return MONARCH_OK;
    return launch_serialized(add_parts_m64_kernel, 2 * (int)(kGradElems / 256), 256, 0, s, (const float *)parts_l, (const float *)parts_r, dL, dR,
                             grid, accumulate);
}

// y = M x, or M^H x, planar complex; e: E tiles of both planes
static int stream_cplx(const void *x, const void *L, const void *R, void *y, int adjoint, void *e, int64_t tokens, unsigned *status, cudaStream_t s)
{
    using namespace tc;
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    const int tiles = (int)tiles_of(tokens), grid = grid_of(kBwdGroups, sms, tokens);
    const size_t plane = (size_t)tokens * kN * 2;
    CUtensorMap tm_w[2], tm_e, tm_x[2], tm_y[2];
    MONARCH_TRY(map_e(&tm_e, e, 2 * tiles, kBwdBlocks));
    MONARCH_TRY(map_w(&tm_w[0], adjoint ? L : R, 2));
    MONARCH_TRY(map_w(&tm_w[1], adjoint ? R : L, 2));
    for (int c = 0; c < 2; ++c) {
        const char *xc = (const char *)x + c * plane, *yc = (const char *)y + c * plane;
        MONARCH_TRY(adjoint ? map_y(&tm_x[c], xc, tokens, kBwdBlocks) : map_t(&tm_x[c], xc, tokens, kBwdBlocks));
        MONARCH_TRY(adjoint ? map_t(&tm_y[c], yc, tokens, kBwdBlocks) : map_y(&tm_y[c], yc, tokens, kBwdBlocks));
    }
    Params p = {};
    p.skip = take_skipped_tile();
    p.status = status;
    p.e_in = (const char *)e;
    p.tiles = tiles;
    MONARCH_TRY(launch_serialized(adjoint ? cplx_kernel<true, true> : cplx_kernel<true, false>, grid, kThreads, kBwdSmem, s, tm_w[0], tm_e, tm_x[0], tm_x[1], p));
    p.skip = -1;
    p.follows = 1;
    p.last = tiles - 1;
    return launch_serialized(adjoint ? cplx_kernel<false, false> : cplx_kernel<false, true>, grid, kThreads, kBwdSmem, s, tm_w[1], tm_e, tm_y[0], tm_y[1], p);
}

// Workspaces: [status][64 KB left out: the counters of kernels that share it stay zero][E tiles ...][parts]
namespace {
constexpr size_t kHead = MONARCH_STATUS_BYTES + 65536;
char *head(const void *ws) { return (char *)ws + kHead; }
}  // namespace

size_t fused_fwd_m64_workspace_bytes(int64_t tokens) { return kHead + tc::e_bytes(tokens); }
const void *fused_fwd_m64_saved_u(const void *fwd_ws) { return head(fwd_ws); }

int fused_fwd_m64(const void *x, const void *L, const void *R, void *y, int64_t tokens, void *ws, cudaStream_t s)
{
    return stream_fwd(x, L, R, nullptr, y, head(ws), tokens, (unsigned *)ws, s);
}
// (the status word is the caller's: `ws` is not initialised)
int fused_fwd_bias_m64(const void *x, const void *L, const void *R, const void *bias, void *y, int64_t tokens, void *ws, void *status,
                       cudaStream_t s)
{
    return stream_fwd(x, L, R, bias, y, head(ws), tokens, (unsigned *)status, s);
}

size_t fused_mlp_fwd_m64_workspace_bytes(int64_t tokens) { return kHead + 2 * tc::e_bytes(tokens); }
int fused_mlp_fwd_m64(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2, void *y,
                      int64_t tokens, void *ws, cudaStream_t s)
{
    using namespace tc;
    if (tokens == 0) return MONARCH_OK;
    char *u = head(ws), *h = u + e_bytes(tokens);
    unsigned *status = (unsigned *)ws;
    if (mlp_prefers_clusters(tokens)) {
        MONARCH_TRY((fwd_on_clusters<false, true, true, true, false>(x, L1, R1, b1, h, nullptr, tokens, false, status, s)));
        return fwd_on_clusters<true, false, true, false, false>(h, L2, R2, b2, y, nullptr, tokens, true, status, s);
    }
    int sms = 0;
    MONARCH_TRY(current_device_sms(&sms));
    MONARCH_TRY((stage1<false, false>(x, R1, nullptr, u, tokens, 0, false, sms, status, s)));
    MONARCH_TRY((stage1<true, true>(u, L1, b1, h, tokens, 1, true, sms, status, s)));
    MONARCH_TRY((stage1<true, false>(h, R2, nullptr, u, tokens, 1, false, sms, status, s)));
    return stage2(u, L2, b2, y, tokens, sms, status, s);
}

size_t fused_bwd_dx_m64_workspace_bytes(int64_t tokens) { return kHead + tc::e_bytes(tokens); }
int fused_bwd_dx_m64(const void *dy, const void *L, const void *R, void *dx, int64_t tokens, void *ws, cudaStream_t s)
{
    return stream_bwd(nullptr, dy, L, R, nullptr, false, dx, nullptr, nullptr, 0, head(ws), nullptr, tokens, (unsigned *)ws, s);
}

size_t fused_bwd_m64_workspace_bytes(int64_t tokens) { return kHead + 2 * tc::e_bytes(tokens) + 2 * tc::max_ranks(tokens) * tc::kGradElems * sizeof(float); }
int fused_bwd_m64(const void *x, const void *dy, const void *L, const void *R, const void *u_saved, void *dx, float *dL, float *dR, int accumulate,
                  int64_t tokens, void *ws, cudaStream_t s)
{
    char *du = head(ws), *u = du + tc::e_bytes(tokens), *parts = u + tc::e_bytes(tokens);
    return stream_bwd(x, dy, L, R, u_saved != nullptr ? u_saved : u, u_saved != nullptr, dx, dL, dR, accumulate, du, parts, tokens, (unsigned *)ws, s);
}

// (E tiles of both planes: a quarter of the workspace that the call asks for at every size)
int fused_cplx_m64(const void *x, const void *L, const void *R, void *y, int adjoint, int64_t tokens, void *ws, cudaStream_t s)
{
    return tokens == 0 ? MONARCH_OK : stream_cplx(x, L, R, y, adjoint, head(ws), tokens, (unsigned *)ws, s);
}

}  // namespace monarch
