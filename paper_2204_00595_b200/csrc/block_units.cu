// The calls that run as one cooperative launch over units of block products (block_units.cuh): which operations a call
// consists of, in which phases, and which tile sizes it runs on.
//
// With the two stages of Section 3.3 as G(W): multiply by the blocks, and P either folded into how a tensor is read or
// written (role kPerm) or not needed (kNat):
//   y  = G(L) G(R) x         kNat by R, then kPerm by L
//   dx = H(R) H(L) dy        kPerm by the blocks of L transposed, then kNat by the blocks of R transposed
//   dL_j = sum_t dy u^T      kPerm;      dR_k = sum_t du x^T      kNat
#include "block_units.cuh"

namespace monarch {
namespace units {
namespace {

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }
size_t esize(int dtype) { return dtype == MONARCH_F32 ? 4 : 2; }
long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }
constexpr int kSms = 148;                              // of the part this library is built for: sizes tiles and splits

// Tile sizes of a launch.  Small: as many CTAs as possible share the weights of a few tokens.  Large: fewer, larger
// units, so that weights and inputs are read less often.
struct Sizes { int TT, ES, LS, KS, TW; };
template <typename T, int M> struct Small { typedef Cfg<T, M, 16, 16, M < 32 ? M : 32, M < 32 ? M : 32> C; };
template <typename T, int M> struct Large { typedef typename Small<T, M>::C C; };
template <> struct Large<bf16, 16> { typedef Cfg<bf16, 16, 64, 16, 16, 16> C; };
template <> struct Large<bf16, 32> { typedef Cfg<bf16, 32, 64, 32, 32, 32> C; };
template <> struct Large<bf16, 64> { typedef Cfg<bf16, 64, 32, 64, 32, 32> C; };
template <> struct Large<float, 32> { typedef Cfg<float, 32, 32, 32, 32, 32, 16> C; };
template <> struct Large<float, 64> { typedef Cfg<float, 64, 32, 64, 64, 64, 16> C; };
template <> struct Large<float, 128> { typedef Cfg<float, 128, 32, 64, 64, 64, 16> C; };

template <typename C> Sizes sizes_of() { return {C::TT, C::ES, C::LS, C::KS, C::TW}; }
template <typename T> Sizes sizes_t(int m, bool large)
{
    switch (m) {
        case 16: return large ? sizes_of<typename Large<T, 16>::C>() : sizes_of<typename Small<T, 16>::C>();
        case 32: return large ? sizes_of<typename Large<T, 32>::C>() : sizes_of<typename Small<T, 32>::C>();
        case 64: return large ? sizes_of<typename Large<T, 64>::C>() : sizes_of<typename Small<T, 64>::C>();
        default: return large ? sizes_of<typename Large<T, 128>::C>() : sizes_of<typename Small<T, 128>::C>();
    }
}
Sizes sizes(int dtype, int m, bool large) { return dtype == MONARCH_F32 ? sizes_t<float>(m, large) : sizes_t<bf16>(m, large); }

// The large tiles once a stage cut into them has a unit for every SM.  fp32: a unit of the large tiles is long (18 us at
// m = 64), so what counts is how full its last wave is; measured, a full wave costs 0.8 of the same work in small tiles plus
// 20 units (m = 64 forward, us, large / small: 500 tokens 37 / 47, 600 tokens 67 / 54, 1000 tokens 74 / 83).
bool use_large(int dtype, int m, int64_t tokens)
{
    const Sizes s = sizes(dtype, m, true);
    const long long units = (m / 8) * (m / s.ES) * ceil_div(tokens, s.TT), waves = ceil_div(units, kSms);
    return dtype == MONARCH_F32 && m > 16 ? 5 * (units + 20) >= 4 * kSms * waves : units >= kSms;
}

constexpr int kMaxSplits = 40;
// Most token ranges of a weight gradient: enough units for every SM, at least four steps in a range.  And a range is summed by one
// accumulator, whose rounding error grows with its length: none is longer than 256 tokens, or tokens / (592 / m) if that is more,
// which is what the staged family sums at a time (staged_simt.cu).  fp32, error of dL for the staged family / at most 16 ranges /
// this: m = 16, 32768 tokens 5.5e-7 / 8.1e-7 / 5.4e-7 (forward + backward 309 -> 180 us), m = 32, 8192 tokens 4.0e-7 / 4.2e-7 /
// 3.0e-7 (256 -> 235 us; 4999 tokens 174 -> 181).
int max_splits(int dtype, int m, int64_t tokens, bool large)
{
    const Sizes s = sizes(dtype, m, large);
    const long long base = (long long)(m / 8) * (m / s.LS) * (m / s.KS), steps = ceil_div(tokens, s.TW);
    long long n = kSms / base;
    if (n > steps / 4) n = steps / 4;
    if (n > kMaxSplits) n = kMaxSplits;
    const long long runs = ceil_div(tokens, 256), most = ceil_div(4 * kSms, m), least = runs < most ? runs : most;
    if (n < least) n = least;
    return n < 1 ? 1 : (int)n;
}
// without empty ranges
int wgrad_splits(int dtype, int m, int64_t tokens, bool large)
{
    const long long steps = ceil_div(tokens, sizes(dtype, m, large).TW), per = ceil_div(steps, max_splits(dtype, m, tokens, large));
    return (int)ceil_div(steps, per);
}
// (for either tiles, and growing with the tokens: a workspace for a batch serves every smaller one)
size_t parts_bytes(int dtype, int m, int64_t tokens)
{
    if (tokens == 0) return 0;
    const int a = max_splits(dtype, m, tokens, false), b = max_splits(dtype, m, tokens, true), s = a > b ? a : b;
    return s > 1 ? up256((size_t)s * m * m * m * sizeof(float)) : 0;
}
size_t act_bytes(int dtype, int m, int64_t tokens) { return up256((size_t)tokens * m * m * esize(dtype)); }

struct Builder {
    Params p;
    Plan plan;
    int m, dtype;
    bool large;
    Sizes sz;

    Builder(int m_, int dtype_, int64_t tokens, void *ws) : m(m_), dtype(dtype_)
    {
        p.n_ops = p.n_phases = 0;
        p.tokens = (int)tokens;
        p.status = (unsigned *)ws;
        large = use_large(dtype, m, tokens);
        sz = sizes(dtype, m, large);
    }
    // a tensor [t][n], or an intermediate, in either role
    View io(const void *q, int perm) const
    {
        const unsigned row = m * m / 8, blk = m / 8;
        return perm ? View{(void *)q, row, 1, blk, 0} : View{(void *)q, row, blk, 1, 0};
    }
    View mid(const void *q, int perm) const
    {
        const unsigned row = m, plane = p.tokens * m;  // of pieces: [j / 8][t][k]
        return perm ? View{(void *)q, row, plane, 1, 1} : View{(void *)q, row, 1, plane, 1};
    }
    Op &add(int kind, int phase, long long units, long long cost)
    {
        Op &o = p.op[p.n_ops];
        o = Op();
        o.kind = kind;
        o.phase = phase;
        o.splits = 1;
        plan.units[p.n_ops] = (int)units;
        // weights are powers of two of a quarter of a stage unit's cost (elements moved)
        const long long quarter = (long long)sz.TT * (m + sz.ES) * 2;
        int sh = 0;
        while (sh < 20 && (quarter << sh) < cost) ++sh;
        plan.shift[p.n_ops] = sh;
        ++p.n_ops;
        if (phase + 1 > p.n_phases) p.n_phases = phase + 1;
        return o;
    }
    Op &stage(int phase, int perm, int trans, View in, const void *w, View out)
    {
        Op &o = add(kStage, phase, (m / 8) * (m / sz.ES) * ceil_div(p.tokens, sz.TT), (long long)sz.TT * (m + sz.ES) * 8);
        o.perm = perm;
        o.trans = trans;
        o.in = in;
        o.w = w;
        o.out = out;
        return o;
    }
    void reduce(int phase, const float *parts, int n, float *sums, long long count, int accumulate)
    {
        Op &o = add(kReduce, phase, ceil_div(count, kReducePer), (long long)kReducePer * (n + 1));
        o.parts = parts;
        o.splits = n;
        o.sums = sums;
        o.count = count;
        o.accumulate = accumulate;
    }
    // the sums in `phase`; where the tokens are split, the parts are added in the next one
    void wgrad(int phase, int perm, View rows, View cols, float *sums, int accumulate, void *parts)
    {
        const int n = wgrad_splits(dtype, m, p.tokens, large);
        Op &o = add(kWgrad, phase, (long long)(m / 8) * (m / sz.LS) * (m / sz.KS) * n,
                    ceil_div(p.tokens, n) * (sz.LS + sz.KS) * 8);
        o.perm = perm;
        o.in = rows;
        o.in2 = cols;
        o.splits = n;
        o.accumulate = accumulate;
        o.sums = n > 1 ? (float *)parts : sums;
        if (n > 1) reduce(phase + 1, (const float *)parts, n, sums, (long long)m * m * m, accumulate);
    }
    void colsum(int phase, View in, float *sums, int accumulate)
    {
        Op &o = add(kColsum, phase, m * m / kColsumCols, (long long)p.tokens * kColsumCols);
        o.in = in;
        o.sums = sums;
        o.accumulate = accumulate;
    }

    int launch(cudaStream_t s) { return dtype == MONARCH_F32 ? launch_t<float>(s) : launch_t<bf16>(s); }

private:
    template <typename T> int launch_t(cudaStream_t s)
    {
        switch (m) {
            case 16: return large ? run<typename Large<T, 16>::C>(s) : run<typename Small<T, 16>::C>(s);
            case 32: return large ? run<typename Large<T, 32>::C>(s) : run<typename Small<T, 32>::C>(s);
            case 64: return large ? run<typename Large<T, 64>::C>(s) : run<typename Small<T, 64>::C>(s);
            case 128: return large ? run<typename Large<T, 128>::C>(s) : run<typename Small<T, 128>::C>(s);
        }
        return MONARCH_ERR_UNSUPPORTED;
    }
    template <typename C> int run(cudaStream_t s)
    {
        static PerDeviceCache resident;                // CTAs that fit on the device at once
        auto kern = units_kernel<C>;
        int fit = resident.get();
        if (fit <= 0) {
            int per_sm = 0, sms = 0;
            MONARCH_TRY(current_device_sms(&sms));
            MONARCH_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem));
            MONARCH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::kThreads, C::kSmem));
            fit = per_sm * sms;
            if (fit <= 0) return MONARCH_ERR_UNSUPPORTED;
            resident.set(fit);
        }
        long long grid = 1;
        for (int ph = 0; ph < p.n_phases; ++ph) {
            long long units = 0;
            for (int o = 0; o < p.n_ops; ++o)
                if (p.op[o].phase == ph) units += plan.units[o];
            if (units > grid) grid = units;
        }
        if (grid > fit) grid = fit;
        for (int ph = 0; ph < p.n_phases; ++ph) {
            long long weight = 0;
            for (int o = 0; o < p.n_ops; ++o)
                if (p.op[o].phase == ph) weight += (long long)plan.units[o] << plan.shift[o];
            plan.share[ph] = weight / grid;
            plan.rest[ph] = weight % grid;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(C::kThreads);
        cfg.dynamicSmemBytes = C::kSmem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;   // all CTAs resident at once: the barriers between phases rely on it
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        MONARCH_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p, plan));
        note_launch();
        return MONARCH_OK;
    }
};

// the status area and the counters of the other kernels, which share the workspace and have to stay zero
constexpr size_t kHead = MONARCH_STATUS_BYTES + 65536;

struct Carve {                                         // buffers from a workspace
    char *at;
    explicit Carve(void *ws) : at((char *)ws + kHead) {}
    void *take(size_t bytes) { void *r = at; at += bytes; return r; }
};

}  // namespace

size_t workspace_bytes(int op, int64_t tokens, int m, int dtype)
{
    const size_t act = act_bytes(dtype, m, tokens), parts = parts_bytes(dtype, m, tokens);
    const size_t sums = up256((size_t)ceil_div(tokens, 16) * m * m * sizeof(float));
    switch (op) {
        case MONARCH_OP_FWD:
        case MONARCH_OP_BWD_DX: return kHead + act;
        case MONARCH_OP_BWD_DW:
        case MONARCH_OP_BWD: return kHead + 2 * act + 2 * parts;
        case MONARCH_OP_MLP_FWD: return kHead + 2 * act;
        case MONARCH_OP_MLP_BWD: return kHead + 6 * act + 4 * parts + sums;
    }
    return 0;
}

void *saved_u(const void *fwd_ws) { return (char *)fwd_ws + kHead; }

int fwd(const void *x, const void *L, const void *R, void *y, int64_t tokens, int m, int dtype, void *u, void *ws, cudaStream_t s)
{
    Builder b(m, dtype, tokens, ws);
    b.stage(0, 0, 0, b.io(x, 0), R, b.mid(u, 0));
    b.stage(1, 1, 0, b.mid(u, 1), L, b.io(y, 1));
    return b.launch(s);
}

int bwd(const void *x, const void *dy, const void *L, const void *R, const void *u_saved, void *dx, float *dL, float *dR,
        int accumulate, int64_t tokens, int m, int dtype, void *ws, cudaStream_t s)
{
    Builder b(m, dtype, tokens, ws);
    const size_t act = act_bytes(dtype, m, tokens), parts = parts_bytes(dtype, m, tokens);
    Carve c(ws);
    void *du = c.take(act);
    b.stage(0, 1, 1, b.io(dy, 1), L, b.mid(du, 1));
    if (dx != nullptr) b.stage(1, 0, 1, b.mid(du, 0), R, b.io(dx, 0));
    if (dL != nullptr) {
        const void *u = u_saved;
        if (u == nullptr) {
            void *own = c.take(act);
            b.stage(0, 0, 0, b.io(x, 0), R, b.mid(own, 0));
            u = own;
        }
        void *part_l = c.take(parts), *part_r = c.take(parts);
        b.wgrad(1, 1, b.io(dy, 1), b.mid(u, 1), dL, accumulate, part_l);
        b.wgrad(1, 0, b.mid(du, 0), b.io(x, 0), dR, accumulate, part_r);
    }
    return b.launch(s);
}

int mlp_fwd(const void *x, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, const void *b2, void *y,
            int64_t tokens, int m, int dtype, void *ws, cudaStream_t s)
{
    Builder b(m, dtype, tokens, ws);
    const size_t act = act_bytes(dtype, m, tokens);
    Carve c(ws);
    void *u = c.take(act), *h = c.take(act);
    b.stage(0, 0, 0, b.io(x, 0), R1, b.mid(u, 0));
    Op &o = b.stage(1, 1, 0, b.mid(u, 1), L1, b.io(h, 1));
    o.bias = b1;
    o.act = kGelu;
    b.stage(2, 0, 0, b.io(h, 0), R2, b.mid(u, 0));
    b.stage(3, 1, 0, b.mid(u, 1), L2, b.io(y, 1)).bias = b2;
    return b.launch(s);
}

// Phases of the chain rule of Section 4 (a = M1 x + b1, h = GELU(a), y = M2 h + b2):
//   0  u1 = R1 x              du2 = L2^T dy          db2
//   1  a, h from u1
//   2  v2 = R2 h              da = R2^T du2 GELU'(a) with its column sums per token tile      dR2
//   3  du1 = L1^T da          dL2                    db1 from those sums
//   4  dx = R1^T du1          dR1, dL1
// (and one phase later each, the sums over token ranges)
int mlp_bwd(const void *x, const void *dy, const void *L1, const void *R1, const void *b1, const void *L2, const void *R2, void *dx,
            float *dL1, float *dR1, float *db1, float *dL2, float *dR2, float *db2, int accumulate, int64_t tokens, int m, int dtype,
            void *ws, cudaStream_t s)
{
    Builder b(m, dtype, tokens, ws);
    const size_t act = act_bytes(dtype, m, tokens), parts = parts_bytes(dtype, m, tokens);
    Carve c(ws);
    void *u1 = c.take(act), *du = c.take(act), *a = c.take(act), *h = c.take(act), *v2 = c.take(act), *da = c.take(act);
    void *part[4] = {c.take(parts), c.take(parts), c.take(parts), c.take(parts)};
    const int tiles = (int)ceil_div(tokens, b.sz.TT), n = m * m;
    float *col = (float *)c.take(0);
    b.stage(0, 0, 0, b.io(x, 0), R1, b.mid(u1, 0));
    b.stage(0, 1, 1, b.io(dy, 1), L2, b.mid(du, 1));
    b.colsum(0, b.io(dy, 0), db2, accumulate);
    Op &act_op = b.stage(1, 1, 0, b.mid(u1, 1), L1, b.io(h, 1));
    act_op.bias = b1;
    act_op.act = kGelu;
    act_op.in2 = b.io(a, 1);
    b.stage(2, 0, 0, b.io(h, 0), R2, b.mid(v2, 0));
    Op &grad_op = b.stage(2, 0, 1, b.mid(du, 0), R2, b.io(da, 0));
    grad_op.act = kGeluGrad;
    grad_op.in2 = b.io(a, 0);
    grad_op.sums = col;
    b.wgrad(2, 0, b.mid(du, 0), b.io(h, 0), dR2, accumulate, part[0]);
    b.stage(3, 1, 1, b.io(da, 1), L1, b.mid(du, 1));
    b.wgrad(3, 1, b.io(dy, 1), b.mid(v2, 1), dL2, accumulate, part[1]);
    b.reduce(3, col, tiles, db1, n, accumulate);
    b.stage(4, 0, 1, b.mid(du, 0), R1, b.io(dx, 0));
    b.wgrad(4, 0, b.mid(du, 0), b.io(x, 0), dR1, accumulate, part[2]);
    b.wgrad(4, 1, b.io(da, 1), b.mid(u1, 1), dL1, accumulate, part[3]);
    return b.launch(s);
}

}  // namespace units
}  // namespace monarch
