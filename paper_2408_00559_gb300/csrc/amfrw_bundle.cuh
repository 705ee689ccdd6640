// AMFR-W2 solver for bundles: up to 32 component grids of one shape, one
// instance per lane.
//
// A batch prices many instances of one shape, so the same component grid
// (levels l) occurs once per instance.  The warp groups of amfrw_solver.cuh
// give a grid its own lanes, one or two nodes each: neighbouring lanes then
// sit on different rows of every axis, and each Outer neighbour, upper face
// and skipped cross term costs the whole warp its instructions (2 700 per
// node and step on the uneven book, about 1 000 of them the method's).  Here
// lane l of every warp of a group holds instance l of the bundle, the group's
// warps share the nodes, and every index, branch and offset is the same for
// the whole warp: blocks of four nodes are evaluated in registers from a
// program built once per bundle (which rows to read, which coefficient rows
// to multiply by; an axis or pair that vanishes at a block is not in it), and
// all values lie as rows of 32 lanes, so every shared-memory access is one
// full row.
//
// Mixed precision: the same operations in the same order as the warp groups'
// solve_item_mixed, so that a price does not depend on which of the two a
// grid went through.  Bound by instruction issue (43 % of the issue slots, 16
// warps per SM; what it waits for is shared-memory latency and the group's
// barriers).  FP64: the pipe is the bound (one warp instruction per 16 cycles
// and SM), so the stencil is kept in the form with the fewest FP64
// instructions that does not cancel on long axes (second differences 2 (X+ - X)
// - (X+ - X-), the gradient shared with the cross terms; neighbour sums with a
// centre coefficient on axes of one and two rows; a term per neighbour that
// exists) and a line is eliminated by one thread (3 instructions a row, against
// 2 log2 P + 3 of a line shared by P lanes).
//
// Measured, the warp groups first: 1024 d=4 level-5 instances in FP64 34.7 ->
// 20.2 ms; the uneven book of 256 (N = 4, 6, 8) in mixed precision 31.4 ->
// 17.4 ms; 512 d=6 level-6 instances in mixed precision, host to host, 88.4 ->
// 49.1 ms; 64 d=6 level-5 instances in FP64 17.5 -> 5.7 ms.
#pragma once
#include "amfrw_solver.cuh"

namespace amfrw {

template <typename V>
__device__ __forceinline__ V bld(const unsigned char* sm, int off)
{
    return *reinterpret_cast<const V*>(sm + off);
}
template <typename V>
__device__ __forceinline__ void bst(unsigned char* sm, int off, V v)
{
    *reinterpret_cast<V*>(sm + off) = v;
}

// Barrier of the warps of one group (ids 1..8: the group's first warp + 1).
__device__ __forceinline__ void bundle_sync(int id, int warps)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(warps * 32) : "memory");
}

// How a source's values enter: increments or Z as one value, Z of the mixed
// precision as an unevaluated pair.
template <typename T, bool PAIR>
struct BundleSrc {
    using V = T;
    __device__ static __forceinline__ V zero() { return T(0); }
    __device__ static __forceinline__ T diff(V a, V b) { return a - b; }
    __device__ static __forceinline__ T val(V a) { return a; }
};
template <>
struct BundleSrc<float, true> {
    using V = float2;
    __device__ static __forceinline__ V zero() { return make_float2(0.f, 0.f); }
    __device__ static __forceinline__ float diff(V a, V b) { return DFSrc::diff(a, b); }
    __device__ static __forceinline__ float val(V a) { return DFSrc::val(a); }
};

// A group's nodes lie in storage order: the axes of the inner block take the
// lowest bits of the node index, the others follow in axis order.  A thread
// takes a block of four nodes at a time (four rows of one axis, or two axes of
// two rows) into registers, so that inside the block every neighbour is
// a register and outside it a whole block of rows lies at one offset: one
// address and one coefficient serve the block's nodes.  Four nodes: with eight
// the unrolled evaluation no longer fits the instruction caches (mixed
// precision, N = 8, level 6: 307 against 205 us a step for a loop over single
// nodes).
// Inner axes NI of a pattern, nodes NB, rows M(a) of inner axis a and bit offset
// S(a) of its row inside the block.
template <int NI_, int M0, int M1, int M2>
struct PatOf {
    static constexpr int NI = NI_, NB = M0 * M1 * M2;
    __host__ __device__ static constexpr int M(int a) { return a == 0 ? M0 : (a == 1 ? M1 : M2); }
    __host__ __device__ static constexpr int log(int m) { return m == 8 ? 3 : (m == 4 ? 2 : (m == 2 ? 1 : 0)); }
    __host__ __device__ static constexpr int S(int a) { return a == 0 ? 0 : (a == 1 ? log(M0) : log(M0) + log(M1)); }
};
template <int PAT>
struct Pat;
template <> struct Pat<kPatSeg> : PatOf<1, 4, 1, 1> {};  // four rows of an axis of 4 rows or more
template <> struct Pat<kPat8> : PatOf<1, 8, 1, 1> {};
template <> struct Pat<kPat42> : PatOf<2, 4, 2, 1> {};
template <> struct Pat<kPat24> : PatOf<2, 2, 4, 1> {};
template <> struct Pat<kPat222> : PatOf<3, 2, 2, 2> {};
template <> struct Pat<kPat4> : PatOf<1, 4, 1, 1> {};
template <> struct Pat<kPat22> : PatOf<2, 2, 2, 1> {};
template <> struct Pat<kPat2> : PatOf<1, 2, 1, 1> {};
template <> struct Pat<kPat1> : PatOf<0, 1, 1, 1> {};

template <int I>
using IntC = std::integral_constant<int, I>;

// Program of a block (int4 records, built once per bundle by bundle_build): a
// head {halo bits, V^2 row, H row, centre row}, {their strides along the
// inner axes}, then for every axis q a region of fixed size:
//   {what | bits, coefficient row, P, Q}   what: 0, 1 inner axis; 2 outside the
//                                          block, at +e_q P, at -e_q Q
//   {outer coefficient row, drift row or -1, pairs, drift strides}
//   per pair with an axis r > q  {A, B, C, D}, {coefficient row, kind, its stride}
// Rows are byte offsets of a row of T; a source of float pairs doubles them.
constexpr int kBlkLo = 1, kBlkTop = 2, kBlkMore = 4;                 // bits of an axis: neighbour below Inner, on the
                                                                      // upper face, rate axis with cross terms
constexpr int kPairIn = 0, kPairOut = 4, kPairOne = 5;               // kPairIn + b: r is the inner axis b
constexpr int kPairLr = 8, kPairLq = 16;                             // neighbours below along r, along q are Inner

// F_0 divided by V^2 at a block of nodes (x: their values), added up in acc.
// Mixed precision (T float): stencil_act2's terms in its order, every product
// fused as there (explicitly: across branches the compiler does not), with
// zeros for Outer neighbours, acc starting as the single-row axes' term.  FP64:
// second differences on axes of four rows or more and outside the block,
// neighbour sums on the block's axes of two rows (acc starts with their and the
// single-row axes' centre term), a term for each neighbour that is not Outer.
template <typename T, bool PAIR, int PAT>
__device__ __forceinline__ void block_F(const unsigned char* sm, int pc, int n, int xs, int at, int zero, int tb, int halos,
                                        const typename BundleSrc<T, PAIR>::V (&x)[Pat<PAT>::NB], T (&acc)[Pat<PAT>::NB])
{
    using P_ = Pat<PAT>;
    using Src = BundleSrc<T, PAIR>;
    using V = typename Src::V;
    constexpr int NB = P_::NB, NI = P_::NI;
    constexpr bool SEG = PAT == kPatSeg, SUM = sizeof(T) == 8;
    constexpr int RB = 32 * sizeof(T), VB = 32 * sizeof(V), SC = PAIR ? 1 : 0;
    // a segment of a longer axis: rows below and above it
    const bool seg_lo = SEG && (halos & 1), seg_last = SEG && !(halos & 2);

    auto load = [&](int off, V (&v)[NB]) {
#pragma unroll
        for (int k = 0; k < NB; ++k) v[k] = bld<V>(sm, xs + (off << SC) + k * VB);
    };
    // the rows beside a segment: 0 below the first row; above the last one is
    // never read (and no row lies beside a block of zeros)
    auto halo = [&](int off, V& hm, V& hp) {
        hm = hp = Src::zero();
        if constexpr (SEG) {
            if (off != zero) {
                if (seg_lo) hm = bld<V>(sm, xs + (off << SC) - VB);
                if (!seg_last) hp = bld<V>(sm, xs + (off << SC) + NB * VB);
            }
        }
    };
    auto row = [](int a, int k) constexpr { return (k >> P_::S(a)) & (P_::M(a) - 1); };
    auto up = [&](int a, int k, const V (&v)[NB], V hp) -> V {
        if (SEG) return k < NB - 1 ? v[k < NB - 1 ? k + 1 : k] : hp;
        return v[(k + (1 << P_::S(a))) & (NB - 1)];
    };
    auto dn = [&](int a, int k, const V (&v)[NB], V hm) -> V {
        if (SEG) return k > 0 ? v[k > 0 ? k - 1 : k] : hm;
        return row(a, k) > 0 ? v[(k - (1 << P_::S(a))) & (NB - 1)] : Src::zero();
    };
    auto top = [&](int a, int k) -> bool { return SEG ? (k == NB - 1 && seg_last) : row(a, k) == P_::M(a) - 1; };

    // p - 2 x + m from g = p - m; without a row below (m = 0), g is not used.
    // (Neighbour sums with a centre coefficient take an operation less, but
    // cancel: they serve the axes of one and two rows.)
    auto second = [](T p, T xv, T g, bool lo) -> T { return lo ? fma(T(2), p - xv, -g) : fma(T(-2), xv, p); };

    // axis q, the inner axis A
    auto inner_axis = [&](auto Ac, int4 h) {
        constexpr int a = decltype(Ac)::value;
        T grad[NB];
        V xm, xp;
        halo(at, xm, xp);
        const int ds = h.z;  // V has one coefficient for all its rows
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const T d = bld<T>(sm, tb + h.y + row(a, k) * ds);
            const V m = dn(a, k, x, xm);
            if constexpr (SUM) {
                const bool lo = SEG ? (k > 0 || seg_lo) : row(a, k) > 0;
                if (top(a, k)) {
                    acc[k] = fma(T(2) * d, SEG ? Src::val(m) - Src::val(x[k]) : Src::val(m), acc[k]);
                    grad[k] = T(0);
                } else {
                    const T p = Src::val(up(a, k, x, xp));
                    grad[k] = lo ? p - Src::val(m) : p;
                    if (SEG) acc[k] = fma(d, second(p, Src::val(x[k]), grad[k], lo), acc[k]);
                    else acc[k] = fma(d, lo ? p + Src::val(m) : p, acc[k]);
                }
            } else {
                const V p = top(a, k) ? m : up(a, k, x, xp);
                const T dp = Src::diff(p, x[k]), dm = Src::diff(x[k], m);
                acc[k] = fma(d, dp - dm, acc[k]);
                grad[k] = dp + dm;
            }
        }
        if (!(h.x & (kBlkMore << 8))) return;
        const int4 e = bld<int4>(sm, pc + 16);
        T in[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) in[k] = T(0);
        int pr = pc + 32;
#pragma unroll 1
        for (int r = e.z; r > 0; --r, pr += 32) {
            const int4 o = bld<int4>(sm, pr), c4 = bld<int4>(sm, pr + 16);
            if (NI > 1 && a == 0 && (c4.y & 7) == kPairIn + 1) {  // the other inner axis
                constexpr int sa = 1, sb = 1 << P_::S(1);
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    if (top(a, k) || row(1, k) == P_::M(1) - 1) continue;
                    const T c = bld<T>(sm, tb + c4.x + row(1, k) * c4.z);
                    const bool la = row(a, k) > 0, lb = row(1, k) > 0;
                    const V pp = x[(k + sa + sb) & (NB - 1)];
                    const V pm = lb ? x[(k + sa - sb) & (NB - 1)] : Src::zero();
                    const V mp = la ? x[(k - sa + sb) & (NB - 1)] : Src::zero();
                    const V mm = la && lb ? x[(k - sa - sb) & (NB - 1)] : Src::zero();
                    in[k] = fma(c, Src::diff(pp, pm) - Src::diff(mp, mm), in[k]);
                }
                continue;
            }
            // differences along axis r at the block's nodes
            const T c = bld<T>(sm, tb + c4.x);
            V P[NB], hm, hp;
            T E[NB], em, ep;
            load(o.x, P);
            halo(o.x, hm, hp);
            if (SUM && !(c4.y & kPairLr)) {
#pragma unroll
                for (int k = 0; k < NB; ++k) E[k] = Src::val(P[k]);
                em = Src::val(hm);
                ep = Src::val(hp);
            } else {
                V Q[NB], gm, gp;
                load(o.y, Q);
                halo(o.y, gm, gp);
#pragma unroll
                for (int k = 0; k < NB; ++k) E[k] = Src::diff(P[k], Q[k]);
                em = Src::diff(hm, gm);
                ep = Src::diff(hp, gp);
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                if (top(a, k)) continue;
                const T eu = SEG ? (k < NB - 1 ? E[k < NB - 1 ? k + 1 : k] : ep) : E[(k + (1 << P_::S(a))) & (NB - 1)];
                if (!SEG && row(a, k) == 0) {
                    in[k] = fma(c, eu, in[k]);
                    continue;
                }
                const T el = SEG ? (k > 0 ? E[k > 0 ? k - 1 : k] : em) : E[(k - (1 << P_::S(a))) & (NB - 1)];
                in[k] = fma(c, eu - el, in[k]);
            }
        }
        const int s0 = e.w & 0xffff, s1 = e.w >> 16;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            if (top(a, k)) continue;
            if (e.y >= 0) in[k] = fma(bld<T>(sm, tb + e.y + row(0, k) * s0 + row(1, k) * s1), grad[k], in[k]);
            acc[k] = fma(bld<T>(sm, tb + e.x + row(a, k) * RB), in[k], acc[k]);
        }
    };

    // axis q outside the block
    auto outer_axis = [&](int4 h) {
        const bool lo = h.x & (kBlkLo << 8);
        const T d = bld<T>(sm, tb + h.y);
        V P[NB], Q[NB];
        T grad[NB];
        if constexpr (SUM) {
            if (lo) load(h.w, Q);
            if (h.x & (kBlkTop << 8)) {
#pragma unroll
                for (int k = 0; k < NB; ++k) acc[k] = fma(T(2) * d, Src::val(Q[k]) - Src::val(x[k]), acc[k]);
                return;
            }
            load(h.z, P);
            if (lo) {
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    grad[k] = Src::val(P[k]) - Src::val(Q[k]);
                    acc[k] = fma(d, second(Src::val(P[k]), Src::val(x[k]), grad[k], true), acc[k]);
                }
            } else {
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    grad[k] = Src::val(P[k]);
                    acc[k] = fma(d, second(grad[k], Src::val(x[k]), T(0), false), acc[k]);
                }
            }
        } else {
            load(h.z, P);  // (on the upper face: the ghost node, the mirror of Q)
            load(h.w, Q);
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const T dp = Src::diff(P[k], x[k]), dm = Src::diff(x[k], Q[k]);
                acc[k] = fma(d, dp - dm, acc[k]);
                grad[k] = dp + dm;
            }
        }
        if (!(h.x & (kBlkMore << 8))) return;
        const int4 e = bld<int4>(sm, pc + 16);
        T in[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) in[k] = T(0);
        int pr = pc + 32;
#pragma unroll 1
        for (int r = e.z; r > 0; --r, pr += 32) {
            const int4 o = bld<int4>(sm, pr), c4 = bld<int4>(sm, pr + 16);
            const int kind = c4.y & 7;
            if (kind == kPairOne) {  // axes of two rows: the upper corner alone
                const T c = bld<T>(sm, tb + c4.x);
                V A[NB];
                load(o.x, A);
#pragma unroll
                for (int k = 0; k < NB; ++k) in[k] = fma(c, Src::val(A[k]), in[k]);
                continue;
            }
            if (kind == kPairOut) {
                const T c = bld<T>(sm, tb + c4.x);
                V A[NB], B[NB];
                T v[NB];
                if constexpr (SUM) {
                    load(o.x, A);
                    if (c4.y & kPairLr) {
                        load(o.y, B);
#pragma unroll
                        for (int k = 0; k < NB; ++k) v[k] = Src::val(A[k]) - Src::val(B[k]);
                    } else {
#pragma unroll
                        for (int k = 0; k < NB; ++k) v[k] = Src::val(A[k]);
                    }
                    if (c4.y & kPairLq) {
                        load(o.z, A);
#pragma unroll
                        for (int k = 0; k < NB; ++k) v[k] -= Src::val(A[k]);
                        if (c4.y & kPairLr) {
                            load(o.w, B);
#pragma unroll
                            for (int k = 0; k < NB; ++k) v[k] += Src::val(B[k]);
                        }
                    }
                } else {
                    V C[NB], D[NB];
                    load(o.x, A);
                    load(o.y, B);
                    load(o.z, C);
                    load(o.w, D);
#pragma unroll
                    for (int k = 0; k < NB; ++k) v[k] = Src::diff(A[k], B[k]) - Src::diff(C[k], D[k]);
                }
#pragma unroll
                for (int k = 0; k < NB; ++k) in[k] = fma(c, v[k], in[k]);
                continue;
            }
            // r is an inner axis
            auto pair = [&](auto Bc) {
                constexpr int b = decltype(Bc)::value;
                if constexpr (b < NI) {
                    V am, ap, bm, bp;
                    halo(h.z, am, ap);
                    halo(h.w, bm, bp);
#pragma unroll
                    for (int k = 0; k < NB; ++k) {
                        if (top(b, k)) continue;
                        const T c = bld<T>(sm, tb + c4.x + row(b, k) * c4.z);
                        if constexpr (SUM) {
                            const T u = SEG ? (k < NB - 1 ? grad[k < NB - 1 ? k + 1 : k] : (lo ? Src::val(ap) - Src::val(bp) : Src::val(ap)))
                                            : grad[(k + (1 << P_::S(b))) & (NB - 1)];
                            if (!SEG && row(b, k) == 0) {
                                in[k] = fma(c, u, in[k]);
                            } else {
                                const T l = SEG ? (k > 0 ? grad[k > 0 ? k - 1 : k] : (lo ? Src::val(am) - Src::val(bm) : Src::val(am)))
                                                : grad[(k - (1 << P_::S(b))) & (NB - 1)];
                                in[k] = fma(c, u - l, in[k]);
                            }
                        } else {
                            const T u = Src::diff(up(b, k, P, ap), dn(b, k, P, am));
                            in[k] = fma(c, u - Src::diff(up(b, k, Q, bp), dn(b, k, Q, bm)), in[k]);
                        }
                    }
                }
            };
            if (NI < 2 || kind == kPairIn) pair(IntC<0>());
            else pair(IntC<1>());
        }
        if (e.y >= 0) {
            const int s0 = e.w & 0xffff, s1 = e.w >> 16;
#pragma unroll
            for (int k = 0; k < NB; ++k)
                in[k] = fma(bld<T>(sm, tb + e.y + row(0, k) * s0 + row(1, k) * s1), grad[k], in[k]);
        }
        const T pw = bld<T>(sm, tb + e.x);
#pragma unroll
        for (int k = 0; k < NB; ++k) acc[k] = fma(pw, in[k], acc[k]);
    };

#pragma unroll 1
    for (int q = 0; q < n; ++q) {
        const int4 h = bld<int4>(sm, pc);
        if (NI > 0 && (h.x & 255) == 0) inner_axis(IntC<0>(), h);
        else if (NI > 1 && (h.x & 255) == 1) inner_axis(IntC<(NI > 1 ? 1 : 0)>(), h);
        else outer_axis(h);
        pc += 32 + 32 * (n - 1 - q);
    }
}

// The directional solves along a group of consecutive axes (at most eight
// rows together), one after the other, for one block of nodes in registers:
// by the explicit inverses (mixed precision, dense_mix's order of terms) or
// Thomas elimination (FP64).  VIN: the last axis is V, so the class (the V
// index) of the rates' lines varies inside the block.
template <typename T, int PAT, bool VIN>
__device__ __forceinline__ void block_solve(const T* lub, const BundleLayout& y, int q0, int cls, T (&x)[Pat<PAT>::NB])
{
    using P_ = Pat<PAT>;
    constexpr int NB = P_::NB, NI = P_::NI;
    constexpr bool DENSE = sizeof(T) == 4;
    auto axis = [&](auto Ac) {
        constexpr int a = decltype(Ac)::value;
        if constexpr (a < NI) {
            constexpr int M = P_::M(a), S = P_::S(a), NC = DENSE ? M * M : 3 * M;
            const int q = q0 + a;
            const T* lu = lub + (y.luoff[q] + (q < y.nr ? cls * NC : 0)) * 32;
            T z[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                if ((k >> S) & (M - 1)) continue;  // k: the line's first node
                const int vr = VIN && a < NI - 1 ? (k >> P_::S(NI - 1)) & (P_::M(NI - 1) - 1) : 0;
                auto c = [&](int e) -> T { return lu[(vr * NC + e) * 32]; };
                if constexpr (DENSE) {
#pragma unroll
                    for (int j = 0; j < M; ++j) {
                        T acc = c(j * M) * x[k + (j << S)];
#pragma unroll
                        for (int e = 1; e < M; ++e) acc = fmaf(c(j * M + e), x[k + ((j ^ e) << S)], acc);
                        z[k + (j << S)] = acc;
                    }
                } else {  // (lower factor, 1/pivot, upper/pivot) per row; row 0 has no lower one
                    z[k] = x[k] * c(1);
#pragma unroll
                    for (int j = 1; j < M; ++j)
                        z[k + (j << S)] = fma(-c(3 * j), z[k + ((j - 1) << S)], x[k + (j << S)]) * c(3 * j + 1);
#pragma unroll
                    for (int j = M - 2; j >= 0; --j)
                        z[k + (j << S)] = fma(-c(3 * j + 2), z[k + ((j + 1) << S)], z[k + (j << S)]);
                }
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) x[k] = z[k];
        }
    };
    axis(IntC<0>());
    axis(IntC<1>());
    axis(IntC<2>());
}

// One group of solves over all its blocks, in place in `dst`.
template <typename T, int PAT, bool VIN>
__device__ __forceinline__ void bundle_group(unsigned char* sm, const T* lub, const BundleLayout& y, int g, int dst, int w,
                                             int W)
{
    using P_ = Pat<PAT>;
    constexpr int NB = P_::NB, NI = P_::NI, RB = 32 * sizeof(T);
    const int q0 = y.gq[g], nb = y.gn[g];
    const unsigned short* blk = reinterpret_cast<const unsigned short*>(sm + y.blk) + y.gblk[g];
    const int st0 = 1 << y.sh[q0], st1 = NI > 1 ? 1 << y.sh[q0 + 1] : 0, st2 = NI > 2 ? 1 << y.sh[q0 + 2] : 0;
#pragma unroll 1
    for (int b = w; b < nb; b += W) {
        const int t0 = blk[b], cls = (t0 >> y.vsh) & y.vmask;
        int t[NB];
        T x[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            t[k] = t0 + (k & (P_::M(0) - 1)) * st0;
            if (NI > 1) t[k] += ((k >> P_::S(1)) & (P_::M(1) - 1)) * st1;
            if (NI > 2) t[k] += ((k >> P_::S(2)) & (P_::M(2) - 1)) * st2;
            x[k] = bld<T>(sm, dst + t[k] * RB);
        }
        block_solve<T, PAT, VIN>(lub, y, q0, cls, x);
#pragma unroll
        for (int k = 0; k < NB; ++k) bst<T>(sm, dst + t[k] * RB, x[k]);
    }
}

// Mixed-precision solves along an axis of 16 rows or more (or the single row
// of a grid of one node): the warp groups' reduction (plog levels of cyclic
// reduction, then at most two rows of Thomas elimination per interleaved
// system), every thread on its own nodes.  The factors of a long axis may lie
// in global scratch, so each level's are loaded before the level ahead of it
// is exchanged.
__device__ __forceinline__ void bundle_long32(unsigned char* sm, int dst, const float* lu, int M, int sh, int plog, int vsh,
                                              int vmask, int L, int w, int W, int bar)
{
    constexpr int NP = 8;  // nodes of a thread at most
    const int S = 2 * plog + 3, P = 1 << plog;
    const int npt = (L + W - 1) / W, t0 = w * npt, t1 = min(L, t0 + npt);
    auto factors = [&](int t) { return lu + ((((t >> vsh) & vmask) * M + ((t >> sh) & (M - 1))) * S) * 32; };
    float al[NP], ga[NP];
    auto fetch = [&](int k) {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (t0 + q >= t1) break;
            const float* rb = factors(t0 + q) + 2 * k * 32;
            al[q] = rb[0];
            ga[q] = rb[32];
        }
    };
    if (plog > 0) fetch(0);
#pragma unroll 1
    for (int k = 0; k < plog; ++k) {
        const int d = 1 << k;
        float v[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int t = t0 + q;
            if (t >= t1) break;
            const int j = (t >> sh) & (M - 1), xa = dst + t * 128;
            const float xm = j >= d ? bld<float>(sm, xa - (d << sh) * 128) : 0.f;
            const float xp = j + d < M ? bld<float>(sm, xa + (d << sh) * 128) : 0.f;
            v[q] = fmaf(-ga[q], xp, fmaf(-al[q], xm, bld<float>(sm, xa)));
        }
        if (k + 1 < plog) fetch(k + 1);
        bundle_sync(bar, W);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (t0 + q >= t1) break;
            bst<float>(sm, dst + (t0 + q) * 128, v[q]);
        }
        bundle_sync(bar, W);
    }
    // a system's first row is one of the P lowest rows; its second lies P above
    const bool two = M > P;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const int t = t0 + q;
        if (t >= t1) break;
        if (((t >> sh) & (M - 1)) >= P) continue;
        const float *rb = factors(t) + 2 * plog * 32, *r1 = rb + P * S * 32;
        const int xa = dst + t * 128, xb = xa + (P << sh) * 128;
        float y = bld<float>(sm, xa) * rb[32];
        if (two) {
            const float y1 = fmaf(-r1[0], y, bld<float>(sm, xb)) * r1[32];
            bst<float>(sm, xb, y1);
            y = fmaf(-rb[64], y1, y);
        }
        bst<float>(sm, xa, y);
    }
}

// FP64 solves along an axis of 16 rows or more (or one row): Thomas
// elimination, a line per warp.
__device__ __forceinline__ void bundle_long64(unsigned char* sm, int dst, const double* lu, int M, int sh, int vsh, int vmask, int L,
                                              int w, int W)
{
    const int nl = L / M, lo = (1 << sh) - 1, st = 256 << sh;
    for (int ln = w; ln < nl; ln += W) {
        const int t0 = (ln & lo) | ((ln >> sh) * (M << sh));
        const double* cb = lu + ((t0 >> vsh) & vmask) * M * 96;
        int xa = dst + t0 * 256;
        double y = bld<double>(sm, xa) * cb[32];
        bst<double>(sm, xa, y);
#pragma unroll 4
        for (int j = 1; j < M; ++j) {
            xa += st;
            cb += 96;
            y = fma(-cb[0], y, bld<double>(sm, xa)) * cb[32];
            bst<double>(sm, xa, y);
        }
#pragma unroll 4
        for (int j = M - 2; j >= 0; --j) {
            xa -= st;
            cb -= 96;
            y = fma(-cb[64], y, bld<double>(sm, xa));
            bst<double>(sm, xa, y);
        }
    }
}

// Payoff part of the interpolation at the spot, sum over the cell's rate
// corners of weight times payoff: axes a.. of the corner tree below a prefix
// (weight, discount product, swap sum).
template <int N, int A>
__device__ __forceinline__ double bundle_corners(const Shape<N>& s, const double* pay, int payoff, const int (&c)[N],
                                                 const double (&w)[N], double wt, double P, double S)
{
    if constexpr (A == N - 1) {
        return wt * fmax(S, 0.0);
    } else {
        double u = 0.0;
#pragma unroll 1
        for (int bit = 0; bit < 2; ++bit) {
            const int o = s.poff[A] + c[A] + bit;
            const double P1 = P * pay[(s.phalf + o) * 32];
            // the caplet's payoff is that of rate 1 alone
            const double S1 = payoff == 0 ? (A == 0 ? pay[o * 32] : S) : fma(pay[o * 32], P1, S);
            u += bundle_corners<N, A + 1>(s, pay, payoff, c, w, wt * (bit ? w[A] : 1.0 - w[A]), P1, S1);
        }
        return u;
    }
}

// The pair and drift coefficients, the line-solve factors and the node
// programs of a bundle.
template <int N, bool MIXED>
__device__ void bundle_build(unsigned char* sm, unsigned char* lub, const BundleLayout& y, const Shape<N>& s, int lane, int w,
                             int W, int bar, double cV, double nudt)
{
    using T = typename std::conditional<MIXED, float, double>::type;
    constexpr int RB = 32 * sizeof(T);
    T* tab = reinterpret_cast<T*>(sm + y.tab) + lane;
    const T* cst = reinterpret_cast<const T*>(sm + y.cst) + lane;
    const double* tabd = reinterpret_cast<const double*>(sm + (MIXED ? y.tabd : y.tab)) + lane;
    T* lu = reinterpret_cast<T*>(lub) + lane;
    // line-solve factors
    if constexpr (MIXED) {
        dense_setup<N, 32>(s, tabd, cV, nudt, lu, w, W);
        // axes of 16 rows or more: pcr_setup's reduction, a row per thread
        for (int i = 0; i < N; ++i) {
            if (((s.skip | s.dense) >> i) & 1) continue;
            const int M = s.M[i], plog = s.plog[i], P = 1 << plog, S = s.luS[i];
            const int ncls = i < N - 1 ? s.M[N - 1] : 1;
            float* A = reinterpret_cast<float*>(sm + y.scr) + lane;  // [2][3][M] rows
            for (int cls = 0; cls < ncls; ++cls) {
                for (int r = w; r < M; r += W) {
                    double a, b, u;
                    matrix_row<N, 32>(s, tabd, cV, nudt, i, cls, r, a, b, u);
                    if (i == s.last && s.skip) {
                        const double f = fold_scale<N, 32>(s, tabd, cV, nudt, i, cls, r);
                        a *= f;
                        b *= f;
                        u *= f;
                    }
                    A[r * 32] = (float)a;
                    A[(M + r) * 32] = (float)b;
                    A[(2 * M + r) * 32] = (float)u;
                }
                bundle_sync(bar, W);
                for (int k = 0; k < plog; ++k) {
                    const int d = 1 << k;
                    const float* X = A + (k & 1) * 3 * M * 32;
                    float* Y = A + ((k + 1) & 1) * 3 * M * 32;
                    for (int r = w; r < M; r += W) {
                        const bool lo = r >= d, hi = r + d < M;
                        const float rb_m = lo ? 1.f / X[(M + r - d) * 32] : 0.f;
                        const float rb_p = hi ? 1.f / X[(M + r + d) * 32] : 0.f;
                        const float al = lo ? X[r * 32] * rb_m : 0.f;
                        const float ga = hi ? X[(2 * M + r) * 32] * rb_p : 0.f;
                        float* row = lu + (s.luoff[i] + (cls * M + r) * S + 2 * k) * 32;
                        row[0] = al;
                        row[32] = ga;
                        const float u_m = lo ? X[(2 * M + r - d) * 32] : 0.f, a_m = lo ? X[(r - d) * 32] : 0.f;
                        const float u_p = hi ? X[(2 * M + r + d) * 32] : 0.f, a_p = hi ? X[(r + d) * 32] : 0.f;
                        Y[(M + r) * 32] = X[(M + r) * 32] - al * u_m - ga * a_p;
                        Y[r * 32] = -al * a_m;
                        Y[(2 * M + r) * 32] = -ga * u_p;
                    }
                    bundle_sync(bar, W);
                }
                const float* X = A + (plog & 1) * 3 * M * 32;
                for (int r = w; r < P; r += W) {
                    float gam = 0.f;
                    for (int q = r; q < M; q += P) {
                        const float inv = 1.f / (X[(M + q) * 32] - X[q * 32] * gam);
                        gam = X[(2 * M + q) * 32] * inv;
                        float* row = lu + (s.luoff[i] + (cls * M + q) * S + 2 * plog) * 32;
                        row[0] = X[q * 32];
                        row[32] = inv;
                        row[64] = gam;
                    }
                }
                bundle_sync(bar, W);
            }
        }
    } else {
        int work = 0, q = -1;
        for (int i = 0; i < N; ++i) {
            if (s.M[i] > 1) ++q;
            if ((s.skip >> i) & 1) continue;
            const int M = s.M[i], ncls = i < N - 1 ? s.M[N - 1] : 1;
            for (int cls = 0; cls < ncls; ++cls) {
                if (work++ % W != w) continue;
                const bool fold = i == s.last && s.skip;
                const double fr = (fold && i < N - 1) ? fold_scale<N, 32>(s, tabd, cV, nudt, i, cls, 0) : 1.0;
                double gam = 0.0;
                double* row = reinterpret_cast<double*>(lu) + ((q >= 0 ? y.luoff[q] : 0) + cls * M * 3) * 32;
                for (int r = 0; r < M; ++r, row += 96) {
                    double a, b, u;
                    matrix_row<N, 32>(s, tabd, cV, nudt, i, cls, r, a, b, u);
                    if (fold) {
                        const double f = i < N - 1 ? fr : fold_scale<N, 32>(s, tabd, cV, nudt, i, cls, r);
                        a *= f;
                        b *= f;
                        u *= f;
                    }
                    const double inv = 1.0 / (b - a * gam);
                    gam = u * inv;
                    row[0] = a;
                    row[32] = inv;
                    row[64] = gam;
                }
            }
        }
    }
    // pair coefficients: cx of the pair times pw of the second (rate) axis
    int pairs = 0;
    for (int q = 0; q < y.nr; ++q) {
        const int i = y.ax[q];
        for (int r = q + 1; r < y.n; ++r) {
            if (pairs++ % W != w) continue;
            const int k = y.ax[r];
            if (r >= y.nr) {
                tab[y.cx[q][r] * 32] = cst[(kOffSm + i) * 32];
            } else {
                const T cx = cst[(kOffRm + upair(i, k)) * 32];
                for (int j = 0; j < s.M[k]; ++j) tab[(y.cx[q][r] + j) * 32] = cx * tab[(s.toff[k] + s.M[k] + j) * 32];
            }
        }
    }
    // drift coefficients S_i g2_i of axis q: one row per index of the rates up to q
    for (int q = 0; q < y.nr; ++q) {
        if (y.dr[q] < 0) continue;
        const int i = y.ax[q];
        T sc = T(0);
        for (int r = 1; r <= i; ++r)
            if (s.M[r] == 1) sc += cst[(kOffRh + ltri(i, r)) * 32] * tab[(s.toff[r] + 2) * 32];
        const T g2 = cst[(kOffG2 + i) * 32];
        for (int t = w; t < y.M[q] * y.qns[q]; t += W) {
            T S = sc;
            for (int r = 0; r <= q; ++r) {
                const int k = y.ax[r];
                if (k < 1) continue;
                const T h = cst[(kOffRh + ltri(i, k)) * 32];
                S += h * tab[(s.toff[k] + 2 * s.M[k] + ((t >> s.sh[k]) & (s.M[k] - 1))) * 32];
            }
            tab[(y.dr[q] + t) * 32] = S * g2;
        }
    }
    if (w == 0) tab[y.cv * 32] = (T)cV;
    if constexpr (!MIXED) {
        // centre coefficients by rate index, of the axes of one row and the
        // block's axes of two
        auto centred = [&](int i) {
            bool c = s.M[i] == 1;
            if (y.pat != kPatSeg)
                for (int b = 0; b < (y.pat == kPat22 ? 2 : (y.pat == kPat2 ? 1 : 0)); ++b) c |= y.ax[y.in[b]] == i;
            return c;
        };
        for (int t = w; t < y.Lr; t += W) {
            double sum = centred(N - 1) ? cV : 0.0;
            for (int i = 0; i < N - 1; ++i)
                if (centred(i)) sum += tab[(s.toff[i] + ((t >> s.sh[i]) & (s.M[i] - 1))) * 32];
            tab[(y.c0 + t) * 32] = -2.0 * sum;
        }
    }
    // base nodes of the solve groups' blocks: the index with the group's bits 0
    unsigned short* blk = reinterpret_cast<unsigned short*>(sm + y.blk);
    for (int g = 0; g < y.ng; ++g) {
        if (y.gpat[g] < 0) continue;
        int mask = 0;
        const int e = g + 1 < y.ng ? y.gq[g + 1] : y.n;
        for (int q = y.gq[g]; q < e; ++q) mask |= (y.M[q] - 1) << y.sh[q];
        for (int b = w * 32 + lane; b < y.gn[g]; b += W * 32) {
            int t = 0, rest = b;
            for (int bit = 1; bit < y.L; bit <<= 1) {
                if (mask & bit) continue;
                if (rest & 1) t |= bit;
                rest >>= 1;
            }
            blk[y.gblk[g] + b] = (unsigned short)t;
        }
    }
    // block programs, a thread per block and axis
    const int nbk = pat_nodes(y.pat), ni = y.pat == kPatSeg || y.pat == kPat2 ? 1 : (y.pat == kPat22 ? 2 : 0);
    const int zero = y.L * RB;
    for (int wk = w * 32 + lane; wk < (y.L / nbk) * (y.n + 1); wk += W * 32) {
        const int b = wk / (y.n + 1), q = wk % (y.n + 1) - 1, t0 = b * nbk, at = t0 * RB;
        int4* blkp = reinterpret_cast<int4*>(sm + y.prog + b * y.pblk);
        auto jrow = [&](int r) { return (t0 >> y.sh[r]) & (y.M[r] - 1); };
        auto rate_row = [&](int e) {  // row in the grid of the rates up to e
            int o = 0;
            for (int r = 0; r <= e; ++r) o += jrow(r) * y.qns[r];
            return o;
        };
        auto strides = [&](int e) {  // what a row of the inner axes adds to it
            int o = 0;
            for (int a = 0; a < ni; ++a)
                if (y.in[a] <= e) o |= (y.qns[y.in[a]] * RB) << (16 * a);
            return o;
        };
        if (q < 0) {
            const int j0 = y.pat == kPatSeg ? jrow(y.in[0]) : 0;
            const int halos = y.pat == kPatSeg ? (j0 > 0 ? 1 : 0) | (j0 + nbk < y.M[y.in[0]] ? 2 : 0) : 0;
            const int rr = rate_row(y.nr - 1);
            int vs = 0;  // V inner: its rows' stride
            for (int a = 0; a < ni; ++a)
                if (y.in[a] >= y.nr) vs |= RB << (16 * a);
            blkp[0] = make_int4(halos, ((t0 >> y.vsh) & y.vmask) * RB, rr * RB, 0);
            blkp[1] = make_int4(vs, strides(y.nr - 1), 0, 0);
            continue;
        }
        int4* rec = blkp + 2;
        for (int r = 0; r < q; ++r) rec += 2 + 2 * (y.n - 1 - r);
        const int in = q == y.in[0] ? 0 : (ni > 1 && q == y.in[1] ? 1 : 2);
        const int j = jrow(q), st = RB << y.sh[q];
        const bool rate = q < y.nr, lo = j > 0, tp = in == 2 && j == y.M[q] - 1, more = rate && !tp;
        const int bits = (lo ? kBlkLo : 0) | (tp ? kBlkTop : 0) | (more ? kBlkMore : 0);
        const int below = lo ? at - st : zero;
        if (in < 2) rec[0] = make_int4(in | (bits << 8), (y.qd[q] + j * y.qds[q]) * RB, y.qds[q] * RB, 0);
        else rec[0] = make_int4(in | (bits << 8), (y.qd[q] + j * y.qds[q]) * RB, tp ? below : at + st, below);
        if (!more) continue;
        int np = 0;
        for (int r = q + 1; r < y.n; ++r) {
            const int rin = r == y.in[0] ? 0 : (ni > 1 && r == y.in[1] ? 1 : 2);
            const int jr = jrow(r), sr = RB << y.sh[r], cs = r < y.nr ? RB : 0;
            if (rin == 2 && jr == y.M[r] - 1) continue;  // on its upper face: no cross term
            const bool lr = jr > 0;
            int4* p = rec + 2 + 2 * np++;
            int kind = kPairIn + rin;
            if (rin == 2) {
                if (in < 2) {
                    kind = kPairOut | (lr ? kPairLr : 0);
                    p[0] = make_int4(at + sr, lr ? at - sr : zero, 0, 0);
                } else {
                    kind = (lr || lo ? kPairOut : kPairOne) | (lr ? kPairLr : 0) | (lo ? kPairLq : 0);
                    p[0] = make_int4(at + st + sr, lr ? at + st - sr : zero, lo ? at - st + sr : zero, lo && lr ? at - st - sr : zero);
                }
            }
            p[1] = make_int4((y.cx[q][r] + (r < y.nr ? jr : 0)) * RB, kind, cs, 0);
        }
        const int e = q < y.nr ? q : y.nr - 1;
        rec[1] = make_int4((y.qpw[q] + j) * RB, y.dr[q] < 0 ? -1 : (y.dr[q] + rate_row(e)) * RB, np, strides(e));
    }
}

// The F evaluation of one phase at all of the group's blocks: right-hand sides
// into `dst` (and R where the phase keeps them).
template <typename T, int PAT>
__device__ __forceinline__ void bundle_rhs(unsigned char* sm, const BundleLayout& y, int ph, int dst, int lane, int tb, int v2,
                                           T dt, T thdt, T a21dt, T cin, int w, int W)
{
    using P_ = Pat<PAT>;
    constexpr int NB = P_::NB, RB = 32 * sizeof(T);
    constexpr bool MIXED = sizeof(T) == 4;
    const int xl = lane * (int)sizeof(T), n = y.n, zero = y.L * RB;
    auto row = [](int a, int k) constexpr { return (k >> P_::S(a)) & (P_::M(a) - 1); };
#pragma unroll 1
    for (int b = w; b * NB < y.L; b += W) {
        const int t0 = b * NB, o = t0 * RB, pc = y.prog + b * y.pblk;
        const int4 h = bld<int4>(sm, pc), hs = bld<int4>(sm, pc + 16);
        const int vb = v2 + h.y, v0 = hs.x & 0xffff, v1 = hs.x >> 16, r0 = hs.y & 0xffff, r1 = hs.y >> 16;
        auto vv = [&](int k) -> T { return bld<T>(sm, vb + row(0, k) * v0 + row(1, k) * v1); };
        auto rrow = [&](int k) { return h.z + row(0, k) * r0 + row(1, k) * r1; };
        auto own = [&](int base, int k) -> T { return bld<T>(sm, base + xl + o + k * RB); };
        T acc[NB], x[NB];
        if constexpr (MIXED) {
            if (ph == 0) {
                float2 z[NB];
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    z[k] = bld<float2>(sm, y.ZZ + lane * 8 + (t0 + k) * 256);
                    acc[k] = cin * (-2.f * DFSrc::val(z[k]));
                }
                block_F<float, true, PAT>(sm, pc + 32, n, y.ZZ + lane * 8, o, zero, tb, h.x, z, acc);
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    x[k] = dt * vv(k) * (bld<float>(sm, y.H + xl + rrow(k)) + acc[k]);
                    bst<float>(sm, y.R + xl + o + k * RB, x[k]);
                }
            } else {
                const int src = ph == 2 ? y.K1 : y.Kw;
                float z[NB];
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    z[k] = own(src, k);
                    acc[k] = cin * (-2.f * z[k]);
                }
                block_F<float, false, PAT>(sm, pc + 32, n, src + xl, o, zero, tb, h.x, z, acc);
                if (ph == 2) {
#pragma unroll
                    for (int k = 0; k < NB; ++k) {
                        x[k] = fmaf((float)kQ21, z[k], fmaf(a21dt * vv(k), acc[k], own(y.R, k)));
                        bst<float>(sm, y.R + xl + o + k * RB, x[k]);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < NB; ++k) x[k] = fmaf(thdt * vv(k), acc[k], 2.f * own(y.R, k) - z[k]);
                }
            }
        } else {
            const int src = ph == 0 ? y.Z : (ph == 2 ? y.K1 : y.Kw);
            double z[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                z[k] = own(src, k);
                const int r = rrow(k);
                acc[k] = bld<double>(sm, tb + y.c0 * RB + r) * z[k];
                if (ph == 0) acc[k] += bld<double>(sm, y.H + xl + r);
            }
            block_F<double, false, PAT>(sm, pc + 32, n, src + xl, o, zero, tb, h.x, z, acc);
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                if (ph == 0) {
                    x[k] = dt * vv(k) * acc[k];
                    bst<double>(sm, y.R + xl + o + k * RB, x[k]);
                } else if (ph == 2) {
                    x[k] = fma(kQ21, z[k], fma(a21dt * vv(k), acc[k], own(y.R, k)));
                    bst<double>(sm, y.R + xl + o + k * RB, x[k]);
                } else {
                    x[k] = fma(thdt * vv(k), acc[k], fma(2.0, own(y.R, k), -z[k]));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < NB; ++k) bst<T>(sm, dst + o + k * RB, x[k]);
    }
}

// One bundle on W warps (this one is warp w of them).
template <int N, bool MIXED>
__device__ void solve_bundle(const BundleArgs& a, const Bundle bd, int tlog, unsigned char* sm, unsigned char* lug, int base,
                             int lane, int w, int W, int bar)
{
    using T = typename std::conditional<MIXED, float, double>::type;
    constexpr int RB = 32 * sizeof(T);
    BundleLayout& y = *reinterpret_cast<BundleLayout*>(sm + base);
    Shape<N>& s = *reinterpret_cast<Shape<N>*>(sm + base + align16((int)sizeof(BundleLayout)));
    const Item& it = a.items[bd.begin + min(lane, bd.count - 1)];  // lanes past the end repeat the last grid
    const InstDev& P = a.insts[it.inst];
    if (w == 0 && lane == 0) {
        y = bundle_layout(N, it.lv, MIXED, tlog, base);
        // mixed precision: the line-solve split of a warp group of 2^tlog lanes
        make_shape<N>(s, it.lv, MIXED ? tlog : 0, MIXED ? kRowsLogWarp : 24, true, true, false, MIXED, 1 << 30);
    }
    bundle_sync(bar, W);
    unsigned char* lub = y.lu >= 0 ? sm + y.lu : lug;
    const double cV = P.cVb * pow2(2 * s.lv[N - 1]), nudt = P.nu * P.dt;
    // 1. tables and constants, a row per warp at a time
    double* tabd = reinterpret_cast<double*>(sm + (MIXED ? y.tabd : y.tab)) + lane;
    const double* pay = reinterpret_cast<const double*>(sm + y.pay) + lane;
    T* tab = reinterpret_cast<T*>(sm + y.tab) + lane;
    T* cst = reinterpret_cast<T*>(sm + y.cst) + lane;
    build_tables<N, MIXED, 32, T>(s, P, tabd, const_cast<double*>(pay), cst, w, W);
    bundle_sync(bar, W);
    if constexpr (MIXED) {
        for (int q = w; q < y.ntab; q += W) tab[q * 32] = (float)tabd[q * 32];
        bundle_sync(bar, W);
    }
    float cin = 0.f;  // the single-row axes' second differences (build_act's sum)
    if constexpr (MIXED)
        for (int i = 0; i < N; ++i)
            if (s.M[i] == 1) cin += i < N - 1 ? tab[s.toff[i] * 32] : (float)cV;
    // 2. F of the payoff on the rate grid, the payoff's part of the interpolation
    T* H = reinterpret_cast<T*>(sm + y.H) + lane;
    for (int t = w; t < y.Lr; t += W) {
        int j[N];
        decode<N>(s, t, j);
        if constexpr (MIXED) H[t * 32] = payoff_H_fast<N, 32>(s, pay, P.payoff, j, (const float*)tab, (const float*)cst);
        else H[t * 32] = payoff_H<N, 32>(s, pay, P.payoff, j, (const double*)tab, (const double*)cst);
    }
    double u;
    {
        int c[N];
        double wt[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const double sx = P.xs[i] * (double)s.M[i];
            int ci = (int)floor(sx);
            ci = ci > s.M[i] - 1 ? s.M[i] - 1 : ci;
            ci = ci < 0 ? 0 : ci;
            c[i] = ci;
            wt[i] = sx - (double)ci;
        }
        // the first axes' corners are shared among the group's warps
        constexpr int SP = N - 1 < 3 ? N - 1 : 3;
        u = 0.0;
        for (int part = w; part < (1 << SP); part += W) {
            double wl = 1.0, Pl = 1.0, Sl = 0.0;
#pragma unroll
            for (int i = 0; i < SP; ++i) {
                const int bit = (part >> i) & 1, o = s.poff[i] + c[i] + bit;
                wl *= bit ? wt[i] : 1.0 - wt[i];
                Pl *= pay[(s.phalf + o) * 32];
                Sl = P.payoff == 0 ? (i == 0 ? pay[o * 32] : Sl) : fma(pay[o * 32], Pl, Sl);
            }
            u += bundle_corners<N, SP>(s, pay, P.payoff, c, wt, wl, Pl, Sl);
        }
    }
    bundle_build<N, MIXED>(sm, lub, y, s, lane, w, W, bar, cV, nudt);
    bundle_sync(bar, W);
    // 3. Z = 0; the setup's scratch shares this memory
    const int xl = lane * (int)sizeof(T), L = y.L;
    for (int t = w; t < L; t += W) {
        bst<double>(sm, y.Z + t * 256 + lane * 8, 0.0);
        if constexpr (MIXED) bst<float2>(sm, y.ZZ + t * 256 + lane * 8, make_float2(0.f, 0.f));
    }
    if constexpr (MIXED) {
        for (int t = L + w; t < L + 4; t += W) {
            bst<float2>(sm, y.ZZ + t * 256 + lane * 8, make_float2(0.f, 0.f));
            bst<float>(sm, y.K1 + t * 128 + xl, 0.f);
            bst<float>(sm, y.Kw + t * 128 + xl, 0.f);
        }
    }
    const T dt = (T)P.dt, thdt = (T)(P.theta * P.dt), a21dt = (T)kA21 * dt;
    const T* lul = reinterpret_cast<const T*>(lub) + lane;  // (a generic address)
    const int tb = y.tab + xl, v2 = tb + s.toff[N - 1] * RB;
    const int Rl = y.R + xl, Kl = y.Kw + xl, K1l = y.K1 + xl, Zl = y.Z + lane * 8, ZZl = y.ZZ + lane * 8;
    bundle_sync(bar, W);
    // 4. time steps: the four phases of solve_item_mixed
    for (int step = 0; step < a.steps; ++step) {
#pragma unroll 1
        for (int ph = 0; ph < 4; ++ph) {
            const int dst = ph == 1 ? K1l : (ph == 3 ? Rl : Kl);
            switch (y.pat) {
                case kPatSeg: bundle_rhs<T, kPatSeg>(sm, y, ph, dst, lane, tb, v2, dt, thdt, a21dt, (T)cin, w, W); break;
                case kPat22: bundle_rhs<T, kPat22>(sm, y, ph, dst, lane, tb, v2, dt, thdt, a21dt, (T)cin, w, W); break;
                case kPat2: bundle_rhs<T, kPat2>(sm, y, ph, dst, lane, tb, v2, dt, thdt, a21dt, (T)cin, w, W); break;
                default: bundle_rhs<T, kPat1>(sm, y, ph, dst, lane, tb, v2, dt, thdt, a21dt, (T)cin, w, W); break;
            }
            bundle_sync(bar, W);
            const int ng = y.ng > 0 ? y.ng : 1;
#pragma unroll 1
            for (int g = 0; g < ng; ++g) {
                const int pat = y.ng > 0 ? y.gpat[g] : -1;
                if (pat < 0) {  // a longer axis (or the one node of a grid without any)
                    const int q = y.ng > 0 ? y.gq[g] : 0, M = y.ng > 0 ? y.M[q] : 1, sh = y.ng > 0 ? y.sh[q] : 0;
                    const T* lu = lul + (y.ng > 0 ? y.luoff[q] : 0) * 32;
                    const int vmask = q < y.nr ? y.vmask : 0;
                    if constexpr (MIXED) bundle_long32(sm, dst, lu, M, sh, y.ng > 0 ? s.plog[y.ax[q]] : 0, y.vsh, vmask, L, w, W, bar);
                    else bundle_long64(sm, dst, lu, M, sh, y.vsh, vmask, L, w, W);
                } else if (y.gv[g]) {
                    if (pat == kPat42) bundle_group<T, kPat42, true>(sm, lul, y, g, dst, w, W);
                    else if (pat == kPat24) bundle_group<T, kPat24, true>(sm, lul, y, g, dst, w, W);
                    else if (pat == kPat222) bundle_group<T, kPat222, true>(sm, lul, y, g, dst, w, W);
                    else bundle_group<T, kPat22, true>(sm, lul, y, g, dst, w, W);
                } else {
                    switch (pat) {
                        case kPat8: bundle_group<T, kPat8, false>(sm, lul, y, g, dst, w, W); break;
                        case kPat42: bundle_group<T, kPat42, false>(sm, lul, y, g, dst, w, W); break;
                        case kPat24: bundle_group<T, kPat24, false>(sm, lul, y, g, dst, w, W); break;
                        case kPat222: bundle_group<T, kPat222, false>(sm, lul, y, g, dst, w, W); break;
                        case kPat4: bundle_group<T, kPat4, false>(sm, lul, y, g, dst, w, W); break;
                        case kPat22: bundle_group<T, kPat22, false>(sm, lul, y, g, dst, w, W); break;
                        default: bundle_group<T, kPat2, false>(sm, lul, y, g, dst, w, W); break;
                    }
                }
                bundle_sync(bar, W);
            }
        }
        // Z + b1 K1 + b2 K2 (K2 is in R) and its float pair
#pragma unroll 2
        for (int t = w; t < L; t += W) {
            const T k1 = bld<T>(sm, K1l + t * RB), k2 = bld<T>(sm, Rl + t * RB);
            const int o = t * 256;
            bst<double>(sm, Zl + o, fma(kB2, (double)k2, fma(kB1, (double)k1, bld<double>(sm, Zl + o))));
            if constexpr (MIXED)
                bst<float2>(sm, ZZl + o, ff_axpy(ff_axpy(bld<float2>(sm, ZZl + o), (float)kB1, k1), (float)kB2, k2));
        }
        bundle_sync(bar, W);
    }
    // 5. Z at the spot's cell: the corners whose every index is Inner, over
    // the axes with more than one row (a single row is the cell's upper corner)
    {
        double wa[6];
        int ca[6];
        double wf = 1.0;
        int q = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const double sx = P.xs[i] * (double)s.M[i];
            int ci = (int)floor(sx);
            ci = ci > s.M[i] - 1 ? s.M[i] - 1 : ci;
            ci = ci < 0 ? 0 : ci;
            const double wi = sx - (double)ci;
            if (s.M[i] == 1) {
                wf *= wi;
            } else {
#pragma unroll
                for (int z = 0; z < 6; ++z)
                    if (z == q) {
                        wa[z] = wi;
                        ca[z] = ci;
                    }
                ++q;
            }
        }
        for (int corner = w; corner < (1 << y.n); corner += W) {
            double wt = wf;
            int t = 0;
            bool in = true;
#pragma unroll
            for (int z = 0; z < 6; ++z) {
                if (z < y.n) {
                    const int bit = (corner >> z) & 1, jj = ca[z] + bit - 1;
                    wt *= bit ? wa[z] : 1.0 - wa[z];
                    in &= jj >= 0;
                    t += jj << y.sh[z];
                }
            }
            if (in && wt != 0.0) u = fma(wt, bld<double>(sm, Zl + t * 256), u);
        }
    }
    const int red = y.red + lane * 8;
    bst<double>(sm, red + w * 256, u);
    bundle_sync(bar, W);
    if (w == 0 && lane < bd.count) {
        double v = u;
        for (int k = 1; k < W; ++k) v += bld<double>(sm, red + k * 256);
        a.u_out[it.out_idx] = v;
    }
    bundle_sync(bar, W);  // the group's memory is reused by its next bundle
}

// Persistent launch over bundle classes in descending group size: a block's
// eight warps form one group for grids of 64 nodes, two of four warps for the
// rest.  A group takes bundles from its class's counter
// until none is left, then goes on to the next class, splitting where that
// class's groups are smaller.
template <int N, bool MIXED>
__global__ void __launch_bounds__(kBundleThreads, MIXED ? 2 : 1) bundle_kernel(BundleArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_next[kBundleThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int first = 0, W = kBundleThreads / 32;
    int c = 0;
    while (c < a.n_classes) {
        const BundleClass cd = a.classes[c];
        while (W > cd.warps) {  // the group splits in two
            W >>= 1;
            if (warp - first >= W) first += W;
        }
        const int w = warp - first, bar = first + 1;
        if (w == 0 && lane == 0) s_next[first] = atomicAdd(a.queue + cd.qidx, 1);
        bundle_sync(bar, W);
        const int k = s_next[first];
        bundle_sync(bar, W);
        if (k >= cd.count) {
            ++c;
            continue;
        }
        unsigned char* lug = a.lu_scratch + (size_t)(blockIdx.x * 2 + first / 4) * (size_t)a.lu_stride;
        solve_bundle<N, MIXED>(a, a.bundles[cd.begin + k], cd.tlog, smem, lug, first * a.smem_warp, lane, w, W, bar);
    }
}

}  // namespace amfrw
