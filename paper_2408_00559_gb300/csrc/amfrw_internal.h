// Library-internal records shared by the host launcher and the kernels.
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define AMFRW_HD __host__ __device__ __forceinline__
#else
#define AMFRW_HD inline
#endif

namespace amfrw {

constexpr int kMaxDim = 8;
constexpr int kCtaMaxThreads = 256;  // CTA work groups (grids of more than 64 Inner nodes)

// Per-instance parameters on the device (one per pricing problem).
struct InstDev {
    int32_t N, payoff, n_steps, precision;
    int32_t grid_begin, grid_count;
    int32_t bc;          // 0: Neumann upper faces (Sketch 1); 1: Dirichlet rate faces (eq. bound1_0)
    int32_t pad1;
    double alpha[kMaxDim], phi[kMaxDim], tau[kMaxDim], F0[kMaxDim];
    double Fmax[kMaxDim];          // Fmax[N-1] = V^max
    double rho[kMaxDim * kMaxDim];  // rate correlations, leading dimension 8
    double sigma, beta, V0, K, T, discount, theta, nu, dt;
    double pad2;
    // The level-free factors of a grid's constants, computed once per
    // instance: h_i = Fmax_i 2^-l_i exactly, so every constant of a grid is
    // one of these times an exact power of two (the same FP64 value as
    // dividing by the grid's h directly).
    double cVb;                                // sigma^2 / (2 Vmax^2), times 4^l_V
    double dcb[kMaxDim];                       // alpha_a^2 rho_aa / (2 Fmax_a^2), times 4^l_a
    double rmb[kMaxDim * (kMaxDim - 1) / 2];   // rho_ik / (4 Fmax_i Fmax_k), times 2^(l_i + l_k)
    double smb[kMaxDim];                       // sigma phi_i / (4 Fmax_i Vmax), times 2^(l_i + l_V)
    double g2b[kMaxDim];                       // 1 / (2 Fmax_i), times 2^l_i
    double xs[kMaxDim];                        // spot over Fmax: F_i(0) / Fmax_i, V0 / Vmax (times M_i: x*/h_i)
};

// One component grid of one instance: the unit of work of the solver.
struct Item {
    int32_t inst;        // instance index
    int32_t out_idx;     // slot of u_l(x*) in the per-grid output array
    int32_t L;           // Inner nodes prod_i M_i
    int32_t pad0;
    int8_t lv[kMaxDim];  // log2 M_i per axis
    int64_t state_off;   // offset (doubles) of the grid's Inner values in the
                         // state pool, or -1 when the state is not kept
};

// Shared-memory layout of one grid inside its work group.  The host uses it
// to size dynamic shared memory, the device to place the arrays; both call
// this one function so they cannot disagree.
struct Layout {
    int32_t meta, cd, cf, tabd, tabf, pay, lu, Z, ZZ, H, DR, FY, K1, K0, Kw, D, C, scr, total;
    // CTA groups: bytes of the block's slice of global scratch (line-solve
    // factors, and in mixed precision Z and dt F(Y_n) at offsets gZ, gFY)
    int32_t gbytes, gZ, gFY;
    int32_t L, Lp, Lr, ntab, npay, nlu, ncoef;
};

// Per-node coefficients of the difference-array stencil (FP64 warp groups):
// N diagonal, 1 centre, N(N-1)/2 cross, N-2 drift, 1 for dt F(payoff).
AMFRW_HD int node_coefs(int N) { return N + 1 + N * (N - 1) / 2 + (N - 2) + 1; }

// Packed index of the pair (i, k), i < k < 8, and of (i, r), r <= i < 8.
AMFRW_HD int upair(int i, int k) { return i * (2 * kMaxDim - i - 1) / 2 + (k - i - 1); }
AMFRW_HD int ltri(int i, int r) { return i * (i + 1) / 2 + r; }

template <typename T>
struct Consts {
    T cV;                 // sigma^2 / (2 h_V^2)
    T dt, thdt, nudt;     // dt, theta*dt, nu*dt
    T rm[kMaxDim * (kMaxDim - 1) / 2];  // rho_ik / (4 h_i h_k), rate pairs i < k (upair)
    T rh[kMaxDim * (kMaxDim + 1) / 2];  // rho_ir for the drift sums, r <= i (ltri)
    T sm[kMaxDim];                      // sigma phi_i / (4 h_i h_V)
    T g2[kMaxDim];                      // 1 / (2 h_i)
};

// Active axes of a grid (those with more than one Inner row) for the
// mixed-precision stencil, built once per grid in shared memory.
// One active axis: read by the stencil as two 16-byte loads.
struct alignas(16) ActAxis {
    int sh;       // bit offset of j - 1 in the node index t
    int msk;      // M - 1
    int nfm;      // j - 1 of the Neumann face, or -2 (Dirichlet data on the upper face)
    int Sp;       // padded stride
    int toff;     // rate axes: offset of their coefficient tables (d, pw, drift)
    int M;        // rows
    int drift;    // 1: rate axis with a drift term (rates 2..N-1)
    int dslot;    // warp groups: its slot in the per-node drift coefficients
};

struct ActAxes {
    int n;                      // active axes, ascending axis order
    int nr;                     // active rate axes (the first nr of them; V, if active, is last)
    float cinact;               // second-difference coefficients of the inactive axes, summed
    int ns;                     // directional solves of a stage (the axes not folded into another)
    ActAxis rec[kMaxDim];
    int ax[kMaxDim];            // the axis index
    float g2[kMaxDim];          // 1 / (2 h) (drift gradient)
    float sconst[kMaxDim];      // drift sum: the part of the inactive rates
    float cx[kMaxDim][kMaxDim]; // pair (q, r), q < r: rho/(4 h h) (two rates) or sigma phi/(4 h h_V)
    float drh[kMaxDim][kMaxDim];// drift of active rate q: rho for the active rates r <= q
    // the solves in ascending axis order, read as one 8-byte load each:
    // [2q] offset of the axis's factors; [2q + 1] sh | M << 8 | axis << 16 |
    // (rate axis) << 24 | (solved by its explicit inverse) << 25
    alignas(8) int sv[2 * kMaxDim];
};

// Per-grid descriptors the mixed-precision solver keeps in shared memory:
// the grid's shape (10 per-axis arrays and 8 scalars of int) and its active
// axes.  Warp groups hold them in their layout; whole-block groups in a
// static shared array of the kernel.
AMFRW_HD constexpr int32_t align16(int32_t x) { return (x + 15) & ~15; }
AMFRW_HD constexpr int shape_bytes(int N) { return align16(4 * (10 * N + 8)); }
AMFRW_HD constexpr int meta_bytes(int N) { return shape_bytes(N) + align16((int)sizeof(ActAxes)); }
constexpr int kMetaBytesMax = meta_bytes(kMaxDim);

// Work-group kinds.  kBundle: grids of one shape of many instances, one instance
// per lane.  kWarpGroup: a grid of at most 64 Inner nodes on (part of) one warp,
// everything in shared memory.  kCtaGroup: one CTA per grid (FP64: or a cluster
// of them), the grid in shared memory, line-solve factors there or in a global
// scratch slice.  kMemGroup: the same with the whole grid state in a slice of
// global scratch (L2/HBM resident): grids too large for shared memory or, in
// mixed precision, with lines of more than 128 rows.
constexpr int kWarpGroup = 0;
constexpr int kCtaGroup = 1;
constexpr int kMemGroup = 2;
constexpr int kBundle = 3;

// Rows of a line per lane in a line solve: at most 2 for warp groups (grids of
// at most 64 Inner nodes) and 4 for mixed-precision CTA groups (rows held in
// registers; they run two blocks per SM, so 128 registers a thread), hence
// lines of at most 128 rows there; unbounded for global-memory groups and FP64
// CTA groups (rows streamed from memory).
constexpr int kRowsLogWarp = 1;
constexpr int kRowsLogCta = 2;
constexpr int kRowsLogMem = 24;
AMFRW_HD int rows_log(int kind) { return kind == kWarpGroup ? kRowsLogWarp : (kind == kCtaGroup ? kRowsLogCta : kRowsLogMem); }

// Lanes per line (as log2) for the directional solves along an axis with
// 2^mlog rows, on a grid of 2^llog Inner nodes solved by a group of 2^tlog
// threads: enough lanes that the whole group is busy, at most 2^rlog rows per
// lane, at most 32 lanes (one warp) and at most one row per lane.
AMFRW_HD int lanes_log(int mlog, int llog, int tlog, int rlog)
{
    int p = tlog + mlog - llog;
    if (p < mlog - rlog) p = mlog - rlog;
    if (p < 0) p = 0;
    if (p > mlog) p = mlog;
    if (p > 5) p = 5;
    return p;
}

// Values stored per matrix row for an axis solved with 2^plog lanes per line:
// PCR multipliers (alpha, gamma) of each level, then the Thomas factors
// (lower, 1/pivot, upper/pivot) of the reduced interleaved systems.
AMFRW_HD int lu_row_values(int plog) { return 2 * plog + 3; }

// Mixed-precision warp groups hold a grid's values in registers (at most two
// nodes per lane) and solve the lines of an axis of 2..8 rows by the explicit
// inverse of its directional matrix: M values per matrix row, the rows of a
// line exchanged by shuffles.  Their offsets are kept 16-byte aligned for
// vector loads.
constexpr int kDenseMaxRows = 8;
AMFRW_HD bool dense_axis(int kind, bool mixed, int M)
{
    return mixed && kind == kWarpGroup && M >= 2 && M <= kDenseMaxRows;
}

// Rows of axis 0 get one padding slot each (lines along axis 0 then start in
// different banks) when they have at least this many nodes.  Mixed-precision
// CTA groups pad only rows of 4 or more, which keeps a 4096-node grid within
// half an SM's shared memory (two resident CTAs); the others pad every row of
// 2 or more.
AMFRW_HD int pad_rows_min(bool lean) { return lean ? 4 : 2; }

// kind: the work-group kind (FP64: warp groups only; whole blocks have
// f64_layout).  Warp and global-memory groups keep the line-solve factors inside
// the layout; CTA groups in the group's slice of a global scratch array.
// Global-memory groups also get FP64 scratch for the factorisation (three values
// per matrix row of the largest axis).  tlog: log2 of the group's thread count.
AMFRW_HD Layout make_layout(int N, const int8_t* lv, bool mixed, int kind, int tlog)
{
    Layout y{};
    int L = 1, sumM = 0, npay = 0;
    for (int i = 0; i < N; ++i) L <<= lv[i];
    for (int i = 0; i < N - 1; ++i) {
        sumM += 1 << lv[i];
        npay += (1 << lv[i]) + 1;
    }
    const int MV = 1 << lv[N - 1];
    const int M0 = 1 << lv[0];
    const bool lean = mixed && kind == kCtaGroup;
    const int pad = M0 >= pad_rows_min(lean) ? 1 : 0;
    y.L = L;
    y.Lp = L + (pad ? (L >> lv[0]) : 0);
    y.Lr = L >> lv[N - 1];
    y.ntab = 3 * sumM + MV;
    y.npay = 2 * npay;
    int llog = 0;
    for (int i = 0; i < N; ++i) llog += lv[i];
    // Mixed-precision warp groups fold the single-row axes into another
    // axis's solve (all rate axes of one row; the V axis of one row when a
    // rate axis has more) and store no factors for them.
    const bool dense = mixed && kind == kWarpGroup;
    bool rate_rows = false;
    for (int i = 0; i < N - 1; ++i) rate_rows |= lv[i] > 0;
    int nlu = 0;
    for (int i = 0; i < N; ++i) {
        const int rows = (i < N - 1 ? MV : 1) << lv[i];  // classes x rows
        if (dense && lv[i] == 0 && (i < N - 1 || rate_rows)) continue;
        if (dense_axis(kind, mixed, 1 << lv[i])) {
            nlu = (nlu + 3) & ~3;
            nlu += rows << lv[i];
        } else {
            nlu += rows * lu_row_values(lanes_log(lv[i], llog, tlog, rows_log(kind)));
        }
    }
    const bool lu_in = kind != kCtaGroup;
    y.nlu = nlu;
    int o = 0;
    if (mixed) {
        // The FP64 constants and tables serve the per-grid setup only (tables,
        // line-solve factors, F of the payoff); the time loop reads their FP32
        // copies.  They share one region with the time loop's vectors.
        y.meta = o; o = align16(o + (kind == kWarpGroup ? meta_bytes(N) : 0));
        y.cf = o;   o = align16(o + (int)sizeof(Consts<float>));
        y.tabf = o; o = align16(o + 4 * y.ntab);
        y.pay = o;  o = align16(o + 8 * y.npay);
        y.lu = o;   o = align16(o + (lu_in ? 4 * y.nlu : 0));
        y.Z = o;    o = align16(o + (lean ? 0 : 8 * y.Lp));
        y.ZZ = o;   o = align16(o + 8 * y.Lp);
        y.H = o;    o = align16(o + 4 * y.Lr);
        // warp groups: per node, the drift coefficient of every refined rate
        // axis 2..N-1 (it depends on the node only, and the time loop would
        // otherwise re-sum it at every F evaluation)
        int ndrift = 0;
        for (int i = 1; i < N - 1; ++i) ndrift += lv[i] > 0 ? 1 : 0;
        y.DR = o;   o = align16(o + (kind == kWarpGroup ? 4 * ndrift * y.Lp : 0));
        int a = o, b = o;
        y.cd = a;   a = align16(a + (int)sizeof(Consts<double>));
        y.tabd = a; a = align16(a + 8 * y.ntab);
        y.FY = b;   b = align16(b + (lean ? 0 : 4 * y.Lp));
        y.K1 = b;   b = align16(b + 4 * y.Lp);
        y.K0 = b;   b = align16(b + 4 * y.Lp);
        y.Kw = b;   b = align16(b + 4 * y.Lp);
        o = a > b ? a : b;
        y.ncoef = 0;
        y.D = o;
        y.C = o;
    } else {
        y.meta = o;
        y.cd = o;   o = align16(o + (int)sizeof(Consts<double>));
        y.cf = o;
        y.tabd = o; o = align16(o + 8 * y.ntab);
        y.tabf = o;
        y.pay = o;  o = align16(o + 8 * y.npay);
        y.lu = o;   o = align16(o + 8 * y.nlu);
        y.Z = o;    o = align16(o + 8 * y.Lp);
        y.ZZ = o;
        y.H = o;    o = align16(o + 8 * y.Lr);
        y.DR = o;
        y.FY = o;
        y.K1 = o;   o = align16(o + 8 * y.Lp);
        y.K0 = o;   o = align16(o + 8 * y.Lp);
        y.Kw = o;   o = align16(o + 8 * y.Lp);
        // central differences per axis and per-node coefficients
        y.ncoef = node_coefs(N);
        y.D = o;    o = align16(o + 8 * N * y.Lp);
        y.C = o;    o = align16(o + 8 * y.ncoef * y.Lp);
    }
    int rmax = 0;
    for (int i = 0; i < N; ++i) {
        const int rows = (i < N - 1 ? MV : 1) << lv[i];
        rmax = rows > rmax ? rows : rmax;
    }
    y.scr = o;  o = align16(o + (kind == kMemGroup ? 3 * 8 * rmax : 0));
    y.total = o;
    // the global slice of a CTA group: factors, then Z and dt F(Y_n)
    y.gbytes = y.gZ = y.gFY = 0;
    if (lean) {
        int g = (4 * nlu + 255) & ~255;
        y.gZ = g;   g += (8 * y.Lp + 255) & ~255;
        y.gFY = g;  g += (4 * y.Lp + 255) & ~255;
        y.gbytes = g;
    }
    return y;
}

// One grid class of a warp-group launch: grids of one size solved by work
// groups of 2^glog lanes (several groups per warp when glog < 5).
struct ClassDesc {
    int32_t glog, item_begin, item_count, smem_group, qidx, pad;  // qidx: its work counter
};

// Launch-time arguments of the solver kernels.
struct SolveArgs {
    const Item* items;
    int32_t n_items;
    int32_t steps;        // steps to take in this launch
    int32_t flags;        // kLoadState | kStoreState
    int32_t smem_group;   // dynamic shared bytes per work group
    const InstDev* insts;
    double* u_out;        // [n grids] u_l(x*)
    double* state;        // state pool (Inner values of Y), may be null
    int32_t* queue;       // work counter, zero before the launch
    unsigned char* lu_scratch;  // CTA groups: Thomas factors, lu_stride bytes per block
    int64_t lu_stride;
    // warp groups: the classes of this launch, walked in order by every warp
    const ClassDesc* classes;
    int32_t n_classes;
    int32_t smem_warp;    // dynamic shared bytes per warp
    // instances to solve (nonzero entries), or null for all: the FP64
    // re-solve of ill-conditioned mixed-precision instances skips the others
    const int32_t* inst_mask;
    int32_t csize;        // FP64 CTA and global-memory groups: blocks per grid (a cluster)
    int32_t budget;       // FP64 whole-block groups: f64_layout's
};

constexpr int kLoadState = 1;
constexpr int kStoreState = 2;
constexpr int kLeanScratch = 4;  // FP64 global-memory groups: the smallest slices

// FP64 grids on whole blocks (amfrw_f64.cuh): offsets of a grid's arrays.  CTA
// groups keep the vectors the stencil reads (Z, K1, Kw) and the small tables in
// shared memory, then what fits the class's budget of the central differences
// (single blocks), the right-hand sides K0 (clusters: their barriers empty the
// L1 cache), the line-solve factors and the tables by rate index, the rest in
// the slice of global scratch; global-memory groups keep everything there.
constexpr int kF64SmemMax = 224 * 1024;
constexpr int kMaxCluster = 8;

// log2 of the lanes among which the lines of a solve are spread: all warps of
// a block; half of a cluster's, whose lines are short enough by then (65x65
// grid on eight blocks: 1.25 ms with a quarter, 1.04 with half, each before
// factors were loaded ahead).
AMFRW_HD int f64_tlog(int csize, int block)
{
    int c = 0, b = 0;
    while ((2 << c) <= csize) ++c;
    while ((2 << b) <= block) ++b;
    return b + (c > 0 ? c - 1 : 0);
}

struct F64Layout {
    int32_t Lp, diff;
    int32_t cst, tabd, pay, cxt, Z, K1, Kw, D, scr;  // in shared memory (global-memory groups: in the slice)
    int32_t lu, H, dr, K0;                           // in the slice, or (bits of `fast`) in shared memory
    int32_t fast;                                    // 1 lu, 2 H, 4 dr, 8 K0
    int32_t smem;
    int64_t slice;
};

// A cluster splits a grid along its longest axis (the last of equal ones):
// each block owns a slab of its rows.
AMFRW_HD int f64_split(int N, const int8_t* lv)
{
    int x = 0;
    for (int i = 1; i < N; ++i)
        if (lv[i] >= lv[x]) x = i;
    return x;
}
// Whether a block meets only its slab's line classes of an axis: two axes split
// along V, where a line of the rate axis is a class.
AMFRW_HD bool f64_own_classes(int N, const int8_t* lv, int axis, int csize)
{
    return N == 2 && axis == 0 && csize > 1 && f64_split(N, lv) == 1;
}

// budget: shared memory a block of a CTA group may fill; 0 for global-memory
// groups without stored differences.
AMFRW_HD F64Layout f64_layout(int N, const int8_t* lv, int kind, int csize, int block, int budget, bool lean)
{
    F64Layout y{};
    int llog = 0, sumM = 0, npay = 0, ncx = 0;
    for (int i = 0; i < N; ++i) llog += lv[i];
    for (int i = 0; i < N - 1; ++i) {
        sumM += 1 << lv[i];
        npay += (1 << lv[i]) + 1;
        for (int k = i + 1; k < N; ++k) ncx += k < N - 1 ? 1 << lv[k] : 1;
    }
    const int MV = 1 << lv[N - 1], L = 1 << llog, Lr = L >> lv[N - 1];
    y.Lp = L + ((1 << lv[0]) >= pad_rows_min(false) ? L >> lv[0] : 0);
    int ndr = 0, sh = 0, rmax = 0;
    int64_t nlu = 0, nlu_own = 0;  // factor values; those one block of a cluster uses
    for (int i = 0; i < N; ++i) {
        const int rows = (i < N - 1 ? MV : 1) << lv[i];
        rmax = rows > rmax ? rows : rmax;
        // (make_shape's line-solve region: folded axes keep their place)
        const int64_t n = (int64_t)rows * lu_row_values(lanes_log(lv[i], llog, f64_tlog(csize, block), kRowsLogMem));
        nlu += n;
        nlu_own += f64_own_classes(N, lv, i, csize) ? n / csize : n;
        if (i >= 1 && i < N - 1 && lv[i] > 0) ndr += 1 << (sh + lv[i] - lv[0]);
        sh += lv[i];
    }
    const bool mem = kind == kMemGroup;
    int64_t g = 0;  // the slice
    int o = 0;      // shared memory
    auto small = [&](int bytes) {
        if (mem) {
            const int64_t at = g;
            g += (bytes + 15) & ~15;
            return (int32_t)at;
        }
        const int at = o;
        o = align16(o + bytes);
        return (int32_t)at;
    };
    y.cst = small(8 * (int)(sizeof(Consts<double>) / sizeof(double)));
    y.tabd = small(8 * (3 * sumM + MV));
    y.pay = small(8 * 2 * npay);
    y.cxt = small(8 * ncx);
    y.Z = small(8 * y.Lp);
    y.scr = y.Z;  // (at most three vectors: rmax <= L)
    y.K1 = small(8 * y.Lp);
    y.Kw = small(8 * y.Lp);
    const int64_t dbytes = (int64_t)8 * (N - 1) * y.Lp;
    y.diff = mem ? (lean || budget == 0 ? 0 : 1) : (csize == 1 && o + dbytes <= budget ? 1 : 0);
    y.D = y.diff ? small((int)dbytes) : 0;
    // in shared memory while it lasts, else in the slice
    auto rest = [&](int64_t fast_bytes, int64_t bytes, int bit) {
        if (!mem && o + fast_bytes + 16 <= budget) {
            y.fast |= bit;
            return small((int)fast_bytes);
        }
        const int64_t at = g;
        g += (bytes + 15) & ~(int64_t)15;
        return (int32_t)at;
    };
    if (csize > 1) y.K0 = rest((int64_t)8 * y.Lp, (int64_t)8 * y.Lp, 8);
    y.lu = rest(8 * nlu_own, 8 * nlu, 1);
    y.H = rest((int64_t)8 * Lr, (int64_t)8 * Lr, 2);
    y.dr = lean ? 0 : rest((int64_t)8 * ndr, (int64_t)8 * ndr, 4);
    if (csize == 1) y.K0 = rest((int64_t)8 * y.Lp, (int64_t)8 * y.Lp, 8);
    y.smem = o;
    y.slice = (g + 255) & ~(int64_t)255;
    return y;
}

// Bundles (amfrw_bundle.cuh): up to 32 grids of one shape, one instance per
// lane, on a group of warps that share the nodes.
constexpr int kBundleThreads = 256;
constexpr int kBundleLanes = 32;
AMFRW_HD int bundle_warps(int L) { return L >= 64 ? 8 : 4; }

struct Bundle {
    int32_t begin, count;  // its grids: consecutive items of equal levels
};

// Bundles of one grid size in a launch.  tlog: log2 lanes of the warp group
// that would solve one of these grids (it fixes the mixed-precision line
// solves' split, so both give the same prices).
struct BundleClass {
    int32_t warps, begin, count, qidx, tlog, pad;
};

struct BundleArgs {
    const Item* items;
    const InstDev* insts;
    const Bundle* bundles;
    const BundleClass* classes;
    double* u_out;
    int32_t* queue;
    int32_t n_classes, steps;
    int32_t smem_warp;  // dynamic shared bytes per warp
    int32_t lu_stride;  // bytes of lu_scratch per half block
    unsigned char* lu_scratch;
};

// Shared memory a bundle of W warps may take: two blocks per SM in mixed
// precision, one in FP64 (whose pipe eight warps keep busy).
constexpr int kBundleSmemMixed = 112 * 1024;
constexpr int kBundleSmemF64 = 225 * 1024;
AMFRW_HD int bundle_budget(bool mixed, int L)
{
    return ((mixed ? kBundleSmemMixed : kBundleSmemF64) / 8 * bundle_warps(L)) & ~255;
}

// Node patterns of a bundle's grid: how many rows of which axes, in axis order,
// a thread holds in registers.  The F evaluation takes blocks of four nodes
// (four rows of one axis, kPatSeg, or two axes of two rows), the directional
// solves up to eight rows of consecutive axes.
// (pat_nodes: nodes of a block of the F evaluation.)
constexpr int kPat8 = 0, kPat42 = 1, kPat24 = 2, kPat222 = 3, kPat4 = 4, kPat22 = 5, kPat2 = 6, kPat1 = 7, kPatSeg = 8;
AMFRW_HD int pat_nodes(int p) { return p == kPatSeg || p == kPat22 ? 4 : (p == kPat2 ? 2 : 1); }

// A bundle's shared memory.  Values of T (float in mixed precision, double
// otherwise) lie in rows of 32 lanes; entries below are row numbers in the
// coefficient table (rows) or byte offsets.  q numbers the axes with more
// than one row, in axis order (V, if among them, is last).
struct BundleLayout {
    int32_t L, Lr, n, nr;             // nodes, rate nodes, axes, rate axes
    int32_t pat, in[2];               // inner block: pattern, its axes q
    int32_t ax[6], M[6], sh[6];       // axis number, rows, bit offset of its index in storage order
    int32_t qd[6], qds[6], qpw[6];    // second-difference coefficients (row stride 0: one for all), outer coefficients
    int32_t qns[6];                   // stride of the axis in the rate grid (V: 0)
    int32_t cx[6][6], dr[6];          // pair coefficients, drift coefficients (-1: none)
    int32_t ntab, cv, c0;             // rows: build_tables' tables; c_V; (FP64) centre coefficients
    int32_t vsh, vmask;               // V's index in storage order
    // the directional solves of a stage: groups of consecutive axes with at
    // most eight rows together (pattern, first q, blocks, base nodes in blk),
    // or one longer axis (pattern -1)
    int32_t ng, gpat[6], gq[6], gv[6], gn[6], gblk[6];
    int32_t luoff[6];                 // rows of an axis's line-solve factors
    int32_t prog, pblk;               // block programs: offset, bytes per block
    int32_t lu, nlu;                  // factors: offset (-1: in global scratch), bytes
    int32_t blk, tab, H, red, Z, ZZ, K1, Kw, R;
    int32_t cst, tabd, pay, scr;      // setup only, in the vectors' memory
    int32_t total;
};

AMFRW_HD BundleLayout bundle_layout(int N, const int8_t* lv, bool mixed, int tlog, int base)
{
    BundleLayout y{};
    const int rb = mixed ? 128 : 256;
    int sh = 0, sumM = 0, npay = 0, longM = 1;
    int bits[6] = {0, 0, 0, 0, 0, 0}, toff = 0;
    for (int i = 0; i < N; ++i) {
        if (lv[i] > 0) {
            const int q = y.n++;
            y.ax[q] = i;
            y.M[q] = 1 << lv[i];
            bits[q] = lv[i];
            y.qns[q] = i < N - 1 ? 1 << sh : 0;
            y.qd[q] = toff;
            y.qds[q] = 1;
            y.qpw[q] = toff + y.M[q];
            if (i < N - 1) ++y.nr;
        }
        if (i < N - 1) {
            sumM += 1 << lv[i];
            npay += (1 << lv[i]) + 1;
            toff += 3 << lv[i];
        }
        sh += lv[i];
    }
    const int MV = 1 << lv[N - 1], tlg = sh;
    y.L = 1 << sh;
    y.Lr = y.L >> lv[N - 1];
    // the inner block: rates if they can fill it, V only when they cannot; an
    // axis of four rows before a longer one, whose blocks have neighbours
    y.pat = kPat1;
    y.in[0] = y.in[1] = -1;
    for (int pass = 0; pass < 2 && y.pat == kPat1; ++pass) {
        const int m = pass == 0 ? y.nr : y.n;
        int one[6], n1 = 0, seg = -1;
        for (int q = 0; q < m; ++q) {
            if (bits[q] == 1) one[n1++] = q;
            else if (seg < 0 || bits[q] < bits[seg]) seg = q;
        }
        if (seg >= 0) {
            y.pat = kPatSeg;
            y.in[0] = seg;
        } else if (n1 >= 2) {
            y.pat = kPat22;
            y.in[0] = one[0];
            y.in[1] = one[1];
        } else if (pass == 1 && n1 == 1) {
            y.pat = kPat2;
            y.in[0] = one[0];
        }
    }
    const int ni = y.pat == kPat22 ? 2 : (y.pat == kPat1 ? 0 : 1);
    sh = 0;
    for (int a = 0; a < ni; ++a) {
        y.sh[y.in[a]] = sh;
        sh += bits[y.in[a]];
    }
    for (int q = 0; q < y.n; ++q) {
        if (q == y.in[0] || q == y.in[1]) continue;
        y.sh[q] = sh;
        sh += bits[q];
    }
    const bool vact = y.n > y.nr;
    y.vsh = vact ? y.sh[y.n - 1] : 0;
    y.vmask = MV - 1;
    // coefficient rows
    int rows = 3 * sumM + MV;
    y.ntab = rows;
    y.cv = rows++;
    if (vact) {
        y.qd[y.n - 1] = y.cv;
        y.qds[y.n - 1] = 0;
    }
    if (!mixed) {
        y.c0 = rows;
        rows += y.Lr;
    }
    for (int q = 0; q < y.n; ++q) {
        y.dr[q] = -1;
        if (q >= y.nr) continue;
        for (int r = q + 1; r < y.n; ++r) {
            y.cx[q][r] = rows;
            rows += r < y.nr ? y.M[r] : 1;
        }
        if (y.ax[q] >= 1) {
            y.dr[q] = rows;
            rows += y.M[q] * y.qns[q];
        }
    }
    // line-solve factors: the sizes of make_shape's (mixed precision), three
    // values a row (FP64); the folded single-row axes have none
    int nlu = 0, nblk = 0;
    for (int q = 0; q < y.n; ++q) {
        const int M = y.M[q], r = (q < y.nr ? MV : 1) * M;
        const bool dense = mixed && M <= kDenseMaxRows;
        if (dense) nlu = (nlu + 3) & ~3;
        y.luoff[q] = nlu;
        if (dense) nlu += r * M;
        else if (mixed) nlu += r * lu_row_values(lanes_log(bits[q], tlg, tlog, kRowsLogWarp));
        else nlu += r * 3;
        if (M > kDenseMaxRows && M > longM) longM = M;
    }
    if (y.n == 0) nlu = 3;
    for (int q = 0; q < y.n;) {
        const int g = y.ng++;
        y.gq[g] = q;
        int b = bits[q], e = q + 1;
        if (b > 3) {
            y.gpat[g] = -1;
        } else {
            while (e < y.n && b + bits[e] <= 3) b += bits[e++];
            y.gpat[g] = b == 3 ? (e - q == 1 ? kPat8 : (e - q == 3 ? kPat222 : (bits[q] == 2 ? kPat42 : kPat24)))
                               : (b == 2 ? (e - q == 1 ? kPat4 : kPat22) : kPat2);
            y.gn[g] = y.L >> b;
            y.gblk[g] = nblk;
            nblk += y.gn[g];
        }
        y.gv[g] = vact && e == y.n && e - q > 1 ? 1 : 0;  // V and rates in one group
        q = e;
    }
    int o = base + align16((int)sizeof(BundleLayout)) + shape_bytes(N);
    y.blk = o;    o = align16(o + 2 * nblk);
    y.pblk = 16 * (2 + 2 * y.n + y.n * (y.n - 1));
    y.prog = o;   o += y.pblk * (y.L / pat_nodes(y.pat));
    y.tab = o;    o += rb * rows;
    y.H = o;      o += rb * y.Lr;
    y.red = o;    o += 256 * bundle_warps(y.L);
    y.nlu = rb * nlu;
    int x = o;
    // (mixed precision: a block of zeros behind each vector the stencil reads,
    // for Outer neighbours)
    const int Lz = y.L + (mixed ? 4 : 0);
    y.Z = x;      x += 256 * y.L;
    y.ZZ = x;     x += mixed ? 256 * Lz : 0;
    y.K1 = x;     x += rb * Lz;
    y.Kw = x;     x += rb * Lz;
    y.R = x;      x += rb * y.L;
    int p = o;
    y.cst = p;    p += rb * (int)(sizeof(Consts<float>) / sizeof(float));
    y.tabd = p;   p += mixed ? 256 * y.ntab : 0;
    y.pay = p;    p += 256 * 2 * npay;
    y.scr = p;    p += mixed ? 128 * 6 * longM : 0;
    // the factors last, in global scratch when they do not fit
    o = x > p ? x : p;
    y.lu = o - base + y.nlu <= bundle_budget(mixed, y.L) ? o : -1;
    y.total = (o + (y.lu < 0 ? 0 : y.nlu) - base + 255) & ~255;
    return y;
}

// Host-side launchers, one translation unit per dimension N.
using LaunchFn = int (*)(const SolveArgs&, bool mixed, int kind, int block, int grid,
                         size_t smem, void* stream);
int launch_n2(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n3(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n4(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n5(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n6(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n7(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_n8(const SolveArgs&, bool, int, int, int, size_t, void*);
int launch_bundle_n2(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n3(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n4(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n5(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n6(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n7(const BundleArgs&, bool, int, size_t, void*);
int launch_bundle_n8(const BundleArgs&, bool, int, size_t, void*);
using BundleFn = int (*)(const BundleArgs&, bool mixed, int grid, size_t smem, void* stream);
// Occupancy query for the same instantiation (blocks per SM).
int occupancy(int N, bool mixed, int kind, int block, size_t smem);
using OccFn = int (*)(bool mixed, int kind, int block, size_t smem);
int occupancy_n2(bool, int, int, size_t);
int occupancy_n3(bool, int, int, size_t);
int occupancy_n4(bool, int, int, size_t);
int occupancy_n5(bool, int, int, size_t);
int occupancy_n6(bool, int, int, size_t);
int occupancy_n7(bool, int, int, size_t);
int occupancy_n8(bool, int, int, size_t);

}  // namespace amfrw
