// FP64 solver of a grid on whole blocks: in shared memory (CTA groups) or with
// its state in a slice of global scratch (global-memory groups), on one block
// or on a cluster of up to eight.
//
// The FP64 pipe bounds these grids (one warp instruction per 16 cycles and
// SM), so each part is written for the fewest FP64 instructions:
//  - the stencil with pair coefficients and drift coefficients from tables and,
//    where the arrays fit, stored central differences D_k = X(+e_k) - X(-e_k),
//    which give the cross terms, the drift and the second differences
//    2 (X(+e_k) - X) - D_k (N = 4: 33 instructions a node against 60 of the
//    direct form).  Neighbour sums with a centre coefficient would take two
//    fewer, but cancel: on a line of 256 rows 1e-12 of the largest value
//    instead of 1e-15;
//  - F(Y_n + a21 K1) = F(Y_n) + a21 F_0(K1), so every evaluation is of F_0;
//  - a line is shared by as few lanes as keep a block's warps busy (each level
//    of cyclic reduction costs two instructions a row, elimination three), its
//    rows streamed from memory instead of held in registers, so a line may
//    have any length.
// A class with at most half as many grids as SMs gives each a cluster, if every
// one of its grids has enough lines and rows along its longest axis for the
// blocks (a class that holds a grid of one line, as the largest grids of a
// standard combination do, runs a block per grid).  A block owns a slab
// of rows of the longest axis: it evaluates the stencil there and solves the
// other axes' lines, which lie inside the slab; rows at the slab's edges are
// stored into the neighbour's copy too.  Lines along the split axis are shared
// out; their values come from and go back to the owners through distributed
// shared memory.
// A class with more grids than SMs runs one, two or four blocks per SM, each
// with its part of the shared memory (f64_widths in amfrw_api.cu).
// Measured, before this kernel -> now: 65x65 full grid, 20 steps, 4.31 -> 0.95
// ms (eight blocks); 120 grids of 128 nodes, 10 steps, 0.46 -> 0.24 ms; a d=4
// level-12 combination, 8 steps: its 1320 grids in shared memory (the largest of
// 4096 nodes; the rest of the time is shared-memory and FP64 latency with eight
// warps per SM) 13.35 -> 12.5 ms, its five grids in global memory 9.4 -> 5.8.
#pragma once
#include <cooperative_groups.h>

#include "amfrw_solver.cuh"

namespace amfrw {

// x with n bits of value v inserted at bit `at`.
__device__ __forceinline__ int insert_bits(int x, int at, int n, int v)
{
    return (x & ((1 << at) - 1)) | (v << at) | ((x >> at) << (at + n));
}

// A block's share of a grid split over a cluster of 2^c blocks along axis x.
struct Slab {
    int c, x, pos, r;  // pos: bit of the node index where the block number starts; r: this block
    __device__ __forceinline__ int owner(int t) const { return (t >> pos) & ((1 << c) - 1); }
    __device__ __forceinline__ int node(int u) const { return insert_bits(u, pos, c, r); }
};

// The solves along one axis of (I - nu dt A_axis), src into dst, the results
// through put(node, index, value).  get(node, index) reads src; lu: the axis's
// factors from line class cls0 on, per row (alpha, gamma) of each level of
// cyclic reduction, then (lower / pivot, 1 / pivot, upper / pivot).  A lane
// streams its R rows B at a time: an FP64 instruction's result is some tens of
// cycles away and a store waits for it, so the rows of a batch are loaded
// first, computed side by side, and stored last; elimination, the one chain,
// takes a single multiply-add per row each way.  MANY: there are several
// batches, and a batch's rows are loaded while the one before it is computed;
// otherwise B = R.  AHEAD: so are its factors, which pays where they lie in
// global scratch (a line of 16384 rows waited for them at every batch: 4.8 ms a
// step, 2.8 so; one of 4096 rows in shared memory, whose factors do not fit
// there, 0.79, 0.64) and not where they lie in shared memory (a d=3 level-9
// combination, 16 steps: 1.13 ms without, 1.19 with).
template <int N, int B, bool MANY, bool AHEAD, class Get, class Put>
__device__ __forceinline__ void sweep_f64_rows(const Shape<N>& s, int axis, const double* lu, double* dst, const Slab& sl,
                                               int cls0, int tid, int nt, Get get, Put put)
{
    const int M = s.M[axis], plog = s.plog[axis], P = 1 << plog, R = MANY ? M >> plog : B, S = s.luS[axis];
    const int lvA = s.lv[axis], sh = s.sh[axis], Spa = s.Sp[axis];
    const bool cut = axis == sl.x;  // lines through all slabs: shared out
    const int nl = (s.L >> lvA) >> sl.c;
    const int MV1 = s.M[N - 1] - 1, shV = s.sh[N - 1];
    const int lpr = nt >> plog, p = tid & (P - 1), slot = tid >> plog;
    for (int base = 0; base < nl; base += lpr) {
        const int line = base + slot;
        const bool act = line < nl;
        if (__ballot_sync(0xffffffffu, act) == 0) break;  // (lines ascend with the warp: none further on)
        const int ln = act ? line : 0;
        int t0;
        if (cut) t0 = insert_bits((ln << sl.c) | sl.r, sh, lvA, 0);
        else if (sl.pos > sh) t0 = sl.node(insert_bits(ln, sh, lvA, 0));
        else t0 = insert_bits(sl.node(ln), sh, lvA, 0);
        const int J0 = s.padded(t0) + p * Spa;
        const int cls = (axis == N - 1) ? 0 : ((t0 >> shV) & MV1) - cls0;
        const double* tb = lu + (cls * M + p) * S;
        const int PS = P * S, PSp = P * Spa;
        // row q of this lane: of src in the first pass, then of dst
        const int st = P << sh, tp = t0 + (p << sh);
        bool first = true;
        auto in = [&](int q) -> double { return first ? get(tp + q * st, J0 + q * PSp) : dst[J0 + q * PSp]; };
        // factor e of the batch of rows from q on
        auto factors = [&](double (&f)[B], bool on, int q, int e) {
#pragma unroll
            for (int i = 0; i < B; ++i) f[i] = on ? tb[(q + i) * PS + e] : 0.0;
        };
        auto rows = [&](double (&v)[B], bool on, int q) {
#pragma unroll
            for (int i = 0; i < B; ++i) v[i] = on ? in(q + i) : 0.0;
        };
        double x[B];
#pragma unroll 1
        for (int k = 0; k < plog; ++k) {
            const int d = 1 << k;
            const int sm = (p - d) & (P - 1), sp = (p + d) & (P - 1);
            const bool send_prev = p >= P - d, send_next = p < d;
            double prev = 0.0;  // the row before the batch, as it was
            double al[B], ga[B];
            rows(x, act, 0);
            if constexpr (AHEAD || !MANY) {
                factors(al, act, 0, 2 * k);
                factors(ga, act, 0, 2 * k + 1);
            }
#pragma unroll 1
            for (int q0 = 0; q0 < R; q0 += B) {
                double nx[B], na[B], ng[B], v[B];
                nx[0] = 0.0;
                if constexpr (MANY) {
                    const bool more = act && q0 + B < R;
                    rows(nx, more, q0 + B);
                    if constexpr (AHEAD) {
                        factors(na, more, q0 + B, 2 * k);
                        factors(ng, more, q0 + B, 2 * k + 1);
                    }
                }
#pragma unroll
                for (int i = 0; i < B; ++i) {
                    const double vm = shfl(send_prev ? (i > 0 ? x[i > 0 ? i - 1 : 0] : prev) : x[i], sm, P, 0xffffffffu);
                    const double vp = shfl(send_next ? (i < B - 1 ? x[i < B - 1 ? i + 1 : i] : nx[0]) : x[i], sp, P, 0xffffffffu);
                    if constexpr (MANY && !AHEAD) {
                        const double* row = tb + (q0 + i) * PS + 2 * k;
                        al[i] = act ? row[0] : 0.0;
                        ga[i] = act ? row[1] : 0.0;
                    }
                    v[i] = fma(-ga[i], vp, fma(-al[i], vm, x[i]));
                }
                prev = x[B - 1];
                if (act) {
#pragma unroll
                    for (int i = 0; i < B; ++i) dst[J0 + (q0 + i) * PSp] = v[i];
                }
                if constexpr (MANY) {
#pragma unroll
                    for (int i = 0; i < B; ++i) {
                        x[i] = nx[i];
                        if constexpr (AHEAD) {
                            al[i] = na[i];
                            ga[i] = ng[i];
                        }
                    }
                }
            }
            first = false;
        }
        if (act) {
            const int e = 2 * plog;
            double y = 0.0, lo[B], iv[B];
            rows(x, true, 0);
            if constexpr (AHEAD || !MANY) {
                factors(lo, true, 0, e);
                factors(iv, true, 0, e + 1);
            }
#pragma unroll 1
            for (int q0 = 0; q0 < R; q0 += B) {
                double nx[B], nlo[B], niv[B];
                const bool more = MANY && q0 + B < R;
                if constexpr (MANY) {
                    rows(nx, more, q0 + B);
                    if constexpr (AHEAD) {
                        factors(nlo, more, q0 + B, e);
                        factors(niv, more, q0 + B, e + 1);
                    } else {
                        factors(iv, true, q0, e + 1);
                    }
                }
#pragma unroll
                for (int i = 0; i < B; ++i) x[i] *= iv[i];
#pragma unroll
                for (int i = 0; i < B; ++i) {
                    if constexpr (MANY && !AHEAD) lo[i] = tb[(q0 + i) * PS + e];
                    if (i > 0 || q0 > 0) x[i] = fma(-lo[i], y, x[i]);
                    y = x[i];
                }
                if constexpr (MANY) {
                    if (more) {
#pragma unroll
                        for (int i = 0; i < B; ++i) dst[J0 + (q0 + i) * PSp] = x[i];
#pragma unroll
                        for (int i = 0; i < B; ++i) {
                            x[i] = nx[i];
                            if constexpr (AHEAD) {
                                lo[i] = nlo[i];
                                iv[i] = niv[i];
                            }
                        }
                    }
                }
            }
            // back from the last batch, which is still in x
            double up[B];
            if constexpr (AHEAD || !MANY) factors(up, true, R - B, e + 2);
            first = false;
#pragma unroll 1
            for (int q0 = R - B; q0 >= 0; q0 -= B) {
                double nx[B], nup[B];
                if constexpr (MANY) {
                    rows(nx, q0 > 0, q0 - B);
                    if constexpr (AHEAD) factors(nup, q0 > 0, q0 - B, e + 2);
                }
#pragma unroll
                for (int i = B - 1; i >= 0; --i) {
                    if constexpr (MANY && !AHEAD) up[i] = tb[(q0 + i) * PS + e + 2];
                    if (i < B - 1 || q0 + B < R) x[i] = fma(-up[i], y, x[i]);
                    y = x[i];
                }
#pragma unroll
                for (int i = 0; i < B; ++i) put(tp + (q0 + i) * st, J0 + (q0 + i) * PSp, x[i]);
                if constexpr (MANY) {
#pragma unroll
                    for (int i = 0; i < B; ++i) {
                        x[i] = nx[i];
                        if constexpr (AHEAD) up[i] = nup[i];
                    }
                }
            }
        }
    }
}

// fast: the factors lie in shared memory (or, from five axes on, where long lines
// are rare in grids that fit there, may as well).
template <int N, class Get, class Put>
__device__ __forceinline__ void sweep_f64(const Shape<N>& s, int axis, const double* lu, bool fast, double* dst,
                                          const Slab& sl, int cls0, int tid, int nt, Get get, Put put)
{
    const int R = s.M[axis] >> s.plog[axis];
    if (R > 4 && !fast) sweep_f64_rows<N, 4, true, true>(s, axis, lu, dst, sl, cls0, tid, nt, get, put);
    else if (R > 4) sweep_f64_rows<N, 4, true, false>(s, axis, lu, dst, sl, cls0, tid, nt, get, put);
    else if (R == 4) sweep_f64_rows<N, 4, false, false>(s, axis, lu, dst, sl, cls0, tid, nt, get, put);
    else if (R == 2) sweep_f64_rows<N, 2, false, false>(s, axis, lu, dst, sl, cls0, tid, nt, get, put);
    else sweep_f64_rows<N, 1, false, false>(s, axis, lu, dst, sl, cls0, tid, nt, get, put);
}

template <int N, int KIND>
__device__ void solve_item_f64(const SolveArgs& a, const Item& it, unsigned char* smem, unsigned char* slice, int crank,
                               int csize)
{
    namespace cg = cooperative_groups;
    constexpr bool MEM = KIND == kMemGroup;
    const int nt = (int)blockDim.x, tid = (int)threadIdx.x;
    const bool lean = (a.flags & kLeanScratch) != 0;
    const F64Layout y = f64_layout(N, it.lv, KIND, csize, nt, a.budget, lean);
    const InstDev& P = a.insts[it.inst];
    Shape<N> s;
    make_shape<N>(s, it.lv, f64_tlog(csize, nt), kRowsLogMem, true, true, P.bc != 0);
    unsigned char* base = MEM ? slice : smem;  // the vectors and the small tables
    double* cst = reinterpret_cast<double*>(base + y.cst);
    double* tabd = reinterpret_cast<double*>(base + y.tabd);
    double* pay = reinterpret_cast<double*>(base + y.pay);
    double* cxt = reinterpret_cast<double*>(base + y.cxt);
    double* Z = reinterpret_cast<double*>(base + y.Z);
    double* K1 = reinterpret_cast<double*>(base + y.K1);
    double* Kw = reinterpret_cast<double*>(base + y.Kw);
    double* D = reinterpret_cast<double*>(base + y.D);
    double* scr = reinterpret_cast<double*>(base + y.scr);
    auto at = [&](int off, int bit) { return reinterpret_cast<double*>(((y.fast & bit) ? smem : slice) + off); };
    double *lu = at(y.lu, 1), *H = at(y.H, 2), *dr = at(y.dr, 4), *K0 = at(y.K0, 8);
    const bool lu_fast = (y.fast & 1) != 0;
    const int Lp = y.Lp;

    // Shared data of a cluster's blocks: global scratch and the copies of the
    // vectors; the barrier orders both.
    auto csync = [&]() {
        if (csize == 1) {
            __syncthreads();
        } else {
            asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        }
    };
    Slab sl;
    sl.c = 31 - __clz(csize);
    sl.x = f64_split(N, it.lv);
    sl.pos = s.sh[sl.x] + s.lv[sl.x] - sl.c;
    sl.r = crank;
    const int Ln = s.L >> sl.c;  // nodes of this block
    const bool remote = !MEM && csize > 1;
    // value of node t (index J) into its owner's copy of a vector, and into
    // the neighbour's when the row is next to its slab
    auto put = [&](double* X, int t, int J, double v) {
        if (!remote) {
            X[J] = v;
            return;
        }
        const int o = sl.owner(t), e = (t >> s.sh[sl.x]) & ((1 << (s.lv[sl.x] - sl.c)) - 1);  // row within the slab
        *cg::cluster_group::map_shared_rank(X + J, o) = v;
        if (e == 0 && o > 0) *cg::cluster_group::map_shared_rank(X + J, o - 1) = v;
        if (e == (1 << (s.lv[sl.x] - sl.c)) - 1 && o < csize - 1) *cg::cluster_group::map_shared_rank(X + J, o + 1) = v;
    };

    // 1. tables (every block its own copy), constants
    const int rank = crank * nt + tid, gsize = csize * nt;  // over the cluster
    build_tables<N>(s, P, tabd, pay, cst, MEM ? rank : tid, MEM ? gsize : nt);
    if (MEM) csync();
    else __syncthreads();
    const double cV = P.cVb * pow2(2 * s.lv[N - 1]), nudt = P.nu * P.dt;
    // pair coefficients cx[i][k][j_k] (V: one) in cxt
    {
        const int r0 = MEM ? rank : tid, rs = MEM ? gsize : nt;
        int o = 0;
#pragma unroll
        for (int i = 0; i < N - 1; ++i)
#pragma unroll
            for (int k = i + 1; k < N; ++k) {
                if (k < N - 1) {
                    const double cx = cst[kOffRm + upair(i, k)];
                    for (int q = r0; q < s.M[k]; q += rs) cxt[o + q] = cx * tabd[s.toff[k] + s.M[k] + q];
                    o += s.M[k];
                } else {
                    if (r0 == 0) cxt[o] = cst[kOffSm + i];
                    o += 1;
                }
            }
    }
    // drift coefficients by rate index; H = F(G)/V^2
    auto drift = [&](int i, const int (&j)[N]) {
        double S = 0.0;
#pragma unroll
        for (int r = 1; r < N - 1; ++r)
            if (r <= i) S += cst[kOffRh + ltri(i, r)] * tabd[s.toff[r] + 2 * s.M[r] + j[r] - 1];
        return S * cst[kOffG2 + i];
    };
    const bool tab_fast = !MEM && csize > 1;  // every block its own copy
    for (int t = tab_fast ? tid : rank; t < s.Lr; t += tab_fast ? nt : gsize) {
        int j[N];
        decode<N>(s, t, j);
        H[t] = dirichlet_node(s, t) ? 0.0 : payoff_H<N>(s, pay, P.payoff, j, tabd, cst);
    }
    if (!lean) {
        int o = 0;
#pragma unroll
        for (int i = 1; i < N - 1; ++i) {
            if (s.M[i] == 1) continue;
            const int n = 1 << (s.sh[i] + s.lv[i] - s.sh[1]);  // rates 2..i
            for (int t = tab_fast ? tid : rank; t < n; t += tab_fast ? nt : gsize) {
                int j[N];
                decode<N>(s, t << s.sh[1], j);
                dr[o + t] = drift(i, j);
            }
            o += n;
        }
    }
    // line-solve factors: cyclic reduction, then elimination of the systems
    // left, as sweep_f64 applies them; a line class per P lanes
    const bool own0 = lu_fast && f64_own_classes(N, it.lv, 0, csize);
    auto lu_at = [&](int axis) { return axis > 0 && own0 ? s.luoff[axis] >> sl.c : s.luoff[axis]; };
    for (int axis = 0; axis < N; ++axis) {
        if ((s.skip >> axis) & 1) continue;  // folded into the solve along s.last
        const int M = s.M[axis], plog = s.plog[axis], Pl = 1 << plog, R = M >> plog, S = s.luS[axis];
        const int ncls = (axis < N - 1) ? s.M[N - 1] : 1, rows = ncls * M;
        double *sa = scr, *sb = scr + rows, *su = scr + 2 * rows;
        // a cluster's blocks with the factors in shared memory: each computes
        // those it uses; else they share the classes
        const bool own = lu_fast && f64_own_classes(N, it.lv, axis, csize);
        const int nown = own ? ncls >> sl.c : ncls, cls0 = own ? crank * nown : 0;
        const int step = csize > 1 && !lu_fast ? csize : 1, first = step > 1 ? crank : 0;
        const int lpr = (nt >> plog) * step, p = tid & (Pl - 1), slot = (tid >> plog) * step + first;
        const bool fold = axis == s.last && s.skip;
        for (int b0 = 0; b0 < nown; b0 += lpr) {
            const bool act = b0 + slot < nown;
            const int cl = cls0 + (act ? b0 + slot : 0), r0 = cl * M + p;
            double* tb = lu + lu_at(axis) + ((cl - cls0) * M + p) * S;
            if (act)
                for (int q = 0; q < R; ++q) {
                    double ra, rb, ru;
                    matrix_row<N>(s, tabd, cV, nudt, axis, cl, p + Pl * q, ra, rb, ru);
                    if (fold) {
                        const double f = fold_scale<N>(s, tabd, cV, nudt, axis, cl, p + Pl * q);
                        ra *= f;
                        rb *= f;
                        ru *= f;
                    }
                    sa[r0 + Pl * q] = ra;
                    sb[r0 + Pl * q] = rb;
                    su[r0 + Pl * q] = ru;
                }
            for (int k = 0; k < plog; ++k) {
                const int d = 1 << k;
                const int sm = (p - d) & (Pl - 1), sp = (p + d) & (Pl - 1);
                const bool wm = p < d, wp = p + d >= Pl, send_prev = p >= Pl - d, send_next = p < d;
                double pa = 0.0, pb = 1.0, pu = 0.0;  // pre-update values of row q-1 (pb: reciprocal)
                double ca = act ? sa[r0] : 0.0, cb = act ? sb[r0] : 1.0, cu = act ? su[r0] : 0.0, cr = 1.0 / cb;
                for (int q = 0; q < R; ++q) {
                    const bool nx = q + 1 < R;
                    const int rn = r0 + Pl * (q + 1);
                    const double na = (act && nx) ? sa[rn] : 0.0, nb = (act && nx) ? sb[rn] : 1.0;
                    const double nu = (act && nx) ? su[rn] : 0.0, nr = 1.0 / nb;
                    const double a_m = shfl(send_prev ? pa : ca, sm, Pl, 0xffffffffu);
                    const double r_m = shfl(send_prev ? pb : cr, sm, Pl, 0xffffffffu);
                    const double u_m = shfl(send_prev ? pu : cu, sm, Pl, 0xffffffffu);
                    const double a_p = shfl(send_next ? na : ca, sp, Pl, 0xffffffffu);
                    const double r_p = shfl(send_next ? nr : cr, sp, Pl, 0xffffffffu);
                    const double u_p = shfl(send_next ? nu : cu, sp, Pl, 0xffffffffu);
                    const double al = (!wm || q >= 1) ? ca * r_m : 0.0;
                    const double ga = (wp && !nx) ? 0.0 : cu * r_p;
                    if (act) {
                        tb[q * Pl * S + 2 * k] = al;
                        tb[q * Pl * S + 2 * k + 1] = ga;
                        const int rq = r0 + Pl * q;
                        sb[rq] = cb - al * u_m - ga * a_p;
                        sa[rq] = -al * a_m;
                        su[rq] = -ga * u_p;
                    }
                    pa = ca;
                    pb = cr;
                    pu = cu;
                    ca = na;
                    cb = nb;
                    cu = nu;
                    cr = nr;
                }
            }
            double gam = 0.0;
            if (act)
                for (int q = 0; q < R; ++q) {
                    const int rq = r0 + Pl * q;
                    const double inv = 1.0 / (sb[rq] - sa[rq] * gam);
                    gam = su[rq] * inv;
                    double* row = tb + q * Pl * S + 2 * plog;
                    row[0] = sa[rq] * inv;
                    row[1] = inv;
                    row[2] = gam;
                }
        }
        if (MEM) csync();  // the next axis reuses scr
        else __syncthreads();
    }
    csync();
    // 2. Z from the state or zero (the scratch above shares its memory)
    for (int u = tid; u < Ln; u += nt) {
        const int t = sl.node(u);
        double z = 0.0;
        if (a.flags & kLoadState) {
            int j[N];
            decode<N>(s, t, j);
            z = a.state[it.state_off + t] - payoff_at<N>(s, pay, P.payoff, j);
        }
        put(Z, t, s.padded(t), z);
    }
    csync();

    // dt F_0(X) / (dt V^2), plus init, at node t
    const bool diff = y.diff;
    auto eval = [&](const double* X, int t, const int (&j)[N], int J, double init) -> double {
        const double x0 = X[J];
        double f = init, dx[N];  // dx: X(+e_i) - X(-e_i), off the upper face
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (s.M[i] > 1) {
                const bool face = j[i] == s.nf[i];
                double d2;
                if (diff && i > 0) {
                    dx[i] = face ? 0.0 : D[(i - 1) * Lp + J];
                    d2 = fma(2.0, X[face ? J - s.Sp[i] : J + s.Sp[i]] - x0, -dx[i]);
                } else {
                    const double xm = j[i] > 1 ? X[J - s.Sp[i]] : 0.0, xp = face ? xm : X[J + s.Sp[i]];
                    dx[i] = xp - xm;
                    d2 = (xp - x0) + (xm - x0);
                }
                f = fma(i < N - 1 ? tabd[s.toff[i] + j[i] - 1] : cV, d2, f);
            } else {
                // one node, on its upper face: the neighbours are the boundary's zeros
                f = fma(i < N - 1 ? tabd[s.toff[i] + j[i] - 1] : cV, -2.0 * x0, f);
            }
        }
        int o = 0, od = 0;
#pragma unroll
        for (int i = 0; i < N - 1; ++i) {
            const bool on = j[i] != s.nf[i];
            double in = 0.0;
#pragma unroll
            for (int k = i + 1; k < N; ++k) {
                if (on && j[k] != s.nf[k]) {
                    const bool li = j[i] > 1;
                    double m;
                    if (diff) {
                        const double* Dk = D + (k - 1) * Lp + J;
                        m = Dk[s.Sp[i]] - (li ? Dk[-s.Sp[i]] : 0.0);
                    } else {
                        const bool lk = j[k] > 1;
                        const double pp = X[J + s.Sp[i] + s.Sp[k]], pm = lk ? X[J + s.Sp[i] - s.Sp[k]] : 0.0;
                        const double mp = li ? X[J - s.Sp[i] + s.Sp[k]] : 0.0;
                        const double mm = li && lk ? X[J - s.Sp[i] - s.Sp[k]] : 0.0;
                        m = (pp - pm) - (mp - mm);
                    }
                    in = fma(cxt[o + (k < N - 1 ? j[k] - 1 : 0)], m, in);
                }
                o += k < N - 1 ? s.M[k] : 1;
            }
            if (i >= 1 && s.M[i] > 1) {
                const int n = 1 << (s.sh[i] + s.lv[i] - s.sh[1]);
                if (on) in = fma(lean ? drift(i, j) : dr[od + ((t >> s.sh[1]) & (n - 1))], dx[i], in);
                od += n;
            }
            if (on) f = fma(tabd[s.toff[i] + s.M[i] + j[i] - 1], in, f);
        }
        return f;
    };
    // D_k = X(+e_k) - X(-e_k), k >= 1, where read: off the upper face of axis k
    auto differences = [&](const double* X) {
        if (!diff) return;
        for (int u = tid; u < Ln; u += nt) {
            const int t = sl.node(u);
            int j[N];
            decode<N>(s, t, j);
            const int J = s.padded(t);
#pragma unroll
            for (int k = 1; k < N; ++k)
                if (j[k] != s.M[k]) D[(k - 1) * Lp + J] = X[J + s.Sp[k]] - (j[k] > 1 ? X[J - s.Sp[k]] : 0.0);
        }
        csync();
    };
    // the stage's solves, `from` into `to`.  Lines along the split axis read the
    // owners' copies of a vector in shared memory; right-hand sides that found
    // no room there (four vectors of 8192 nodes do not fit) lie in the
    // cluster's one slice and are read directly: only a shared address may be
    // mapped to another block.
    const bool k0_fast = (y.fast & 8) != 0;
    auto solves = [&](const double* from, double* to) {
        const double* src = from;
        for (int ax = 0; ax < N; ++ax) {
            if ((s.skip >> ax) & 1) continue;
            const bool far = remote && ax == sl.x && (src != K0 || k0_fast);
            sweep_f64<N>(
                s, ax, lu + lu_at(ax), !MEM && (lu_fast || N > 4), to, sl, ax == 0 && own0 ? crank * (s.M[N - 1] >> sl.c) : 0, tid, nt,
                [&](int t, int J) -> double {
                    return far ? *cg::cluster_group::map_shared_rank(const_cast<double*>(src) + J, sl.owner(t)) : src[J];
                },
                [&](int t, int J, double v) { put(to, t, J, v); });
            csync();
            src = to;
        }
    };
    const double theta = P.theta;
    const double* v2 = tabd + s.toff[N - 1] - 1;
#pragma unroll 1
    for (int n = 0; n < a.steps; ++n) {
#pragma unroll 1
        for (int ph = 0; ph < 4; ++ph) {
            const double* X = ph == 0 ? Z : (ph == 2 ? K1 : Kw);
            differences(X);
            double* out = ph == 1 ? K1 : K0;  // (its slab's own rows: the solves come first)
            for (int u = tid; u < Ln; u += nt) {
                const int t = sl.node(u), J = s.padded(t);
                double x = 0.0;
                if (!dirichlet_node(s, t)) {
                    int j[N];
                    decode<N>(s, t, j);
                    const double vd = v2[j[N - 1]] * P.dt;
                    const double f = eval(X, t, j, J, ph == 0 ? H[t & (s.Lr - 1)] : 0.0);
                    if (ph == 0) x = vd * f;
                    else if (ph == 2) x = fma(kQ21, X[J], fma(kA21 * vd, f, K0[J]));
                    else x = fma(theta * vd, f, fma(2.0, K0[J], -X[J]));
                }
                out[J] = x;
            }
            csync();
            if (ph == 1) solves(K1, K1);
            else solves(K0, Kw);
        }
        for (int u = tid; u < Ln; u += nt) {
            const int t = sl.node(u), J = s.padded(t);
            put(Z, t, J, fma(kB2, Kw[J], fma(kB1, K1[J], Z[J])));
        }
        csync();
    }
    // 3. state and interpolation
    if (a.flags & kStoreState) {
        for (int u = tid; u < Ln; u += nt) {
            const int t = sl.node(u);
            int j[N];
            decode<N>(s, t, j);
            a.state[it.state_off + t] = payoff_at<N>(s, pay, P.payoff, j) + Z[s.padded(t)];
        }
    }
    if (remote && crank == 0) {  // the cell may lie in any slab
        for (int t = tid; t < s.L; t += nt)
            if (sl.owner(t) != 0) Z[s.padded(t)] = *cg::cluster_group::map_shared_rank(Z + s.padded(t), sl.owner(t));
        __syncthreads();
    }
    if (crank == 0) interp_spot<N, false>(s, P, pay, Z, a.u_out + it.out_idx, tid, nt, 0xffffffffu);
    csync();  // the memory is reused by the next grid
}

}  // namespace amfrw
