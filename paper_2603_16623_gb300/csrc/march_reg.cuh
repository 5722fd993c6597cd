// march_reg.cuh -- the AB2 march of beam-grid wakes (and of FP64 wakes of a
// given block size) and the RK4 march with a wake's rings in registers.
//
// The chain and the formulas are those of march.cuh and march_rk4.cuh, for
// shapes of up to 4 rings per thread; the marches there, which keep every
// per-ring value in global memory, serve shapes of more.  They spent their
// time on that: ~25 strided reads and writes of per-ring values per ring and
// evaluation, each phase waiting for the last one's through L1 or, after a
// cluster barrier, L2 (long scoreboard first in their profiles), the
// logarithm, the weights and the quotients hA / r taken two to four times.
// Here a thread loads its rings once (again after a re-sort), keeps what only
// it reads in registers, and exchanges with the others
//   - through one-barrier block scans and one fold per cluster exchange: the
//     sums of w and w ln rho; the d_zeta psi sum with the solve's matrices
//     (both depend on psi only); the Green's sums;
//   - two neighbours' edges: the regular solution walked to the end of the
//     rings before (R at its first region; with ring_jump.cuh's products the
//     thread's own) and the next thread's first region (a, b), by shuffle,
//     shared memory, or global memory between blocks;
//   - region tables and radii in global memory, only in slices with beam
//     particles to serve (stage 1 of RK4).
// Crossed rings move to counted ranks (rank_sort.cuh) instead of through one
// block's bitonic network.  The grids' node charges are summed by a warp per
// species (one thread took 53k of a slice's 183k cycles for 33 nodes: FP64
// quotients one after the other) and kept in shared memory, and a ring beyond
// a grid takes one FP64 quotient.
// Measured on GB300, 24 wakes of 500-8000 rings in one batch: RK4 190 -> 89
// us per slice, grids of 32 cells 101 -> 40.  Above 4 rings per thread the
// registers do not hold a thread's values (2 at 512 threads).
#pragma once

#include <type_traits>

#include "march_rk4.cuh"
#include "rank_sort.cuh"

namespace gbwake {

constexpr int kGmWarps = 16;

// a x b rounded (not contracted into a sum), and the fused product sum
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float acc_hi(ff a) { return a.hi; }
__device__ __forceinline__ double acc_hi(double a) { return a; }

// Shared memory of the evaluation (one use of each part per evaluation, so
// that nothing is written again before a later barrier).
template <class P>
struct GmShared {
    using R = typename P::R;
    using A = typename P::A;
    Pair<A> w[kGmWarps], g[kGmWarps];
    SumMats<A, R> m[kGmWarps];
    Pair<A> pre_w, tot_w, pre_g, tot_g;
    A pre_t, tot_t;
    Mat2<R> pre_f, pre_r;
    R edge_r[2][kGmWarps];  // R at the end of each warp
    R edge_a[2][kGmWarps];  // a, b at the start of each warp
};

// the fold of the blocks' totals in rank order (reversed for REV), as every
// thread of the marches of march.cuh takes it: before this block, and of all
template <bool REV, class T, class V, class Op, class Get>
__device__ __forceinline__ void gm_fold(const WakeCtas& C, const V* buf, T ident, Op op, Get get, T& pre, T& tot) {
    pre = ident;
    tot = ident;
    for (int i = 0; i < C.size; ++i) {
        const int r = REV ? C.size - 1 - i : i;
        if (r == C.rank) pre = tot;
        tot = op(tot, get(C.slot(buf, r)));
    }
}

// K values at sorted positions [p0, p0 + np) of a global array
template <int K, class V>
__device__ __forceinline__ void load_rings(const V* a, int p0, int np, V (&v)[K], V fill) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = k < np ? a[p0 + k] : fill;
}

// The wake's column, as both marches take it.
template <class P>
struct Column {
    using R = typename P::R;
    using A = typename P::A;
    R rmax, half_n, quarter_n;
    A Imax, c0;
    __device__ __forceinline__ explicit Column(const WakeDev<P>& W) {
        const double d = W.density, rm = W.rho_max;
        rmax = (R)rm;
        half_n = (R)(0.5 * d);
        quarter_n = (R)(0.25 * d);
        Imax = acc_from_d(0.5 * d * rm * rm, A());
        c0 = acc_from_d(0.25 * d * rm * rm - 0.5 * d * rm * rm * log(rm), A());
    }
};

// Eqs. b_coeffs_2, 3: the ring sources B and C of the B_theta^(p) system
template <class R>
__device__ __forceinline__ void ring_sources(R w, R r, R u, R pb, R g, R dpr, R dpz, R bb, R& Bc, R& Cc) {
    const R wr = w / r, pb2 = pb * pb;
    Bc = -wr * g * dpr / pb2 + wr * bb / pb + (w / (r * r)) * u * u / pb2 + wr * u * u * dpr / (pb2 * pb) -
         wr * u * dpz / pb2;
    Cc = -wr * (g / pb - (R)1 - u * u / pb2);
}

// The jump matrices of a thread's rings multiplied up (Mf, later rings on the
// left) and their inverses multiplied back (Mb), as they are or less the
// identity (Op, ring_jump.cuh); Ac: Eq. b_coeffs_1, m01 = Ac / (2 r).
template <int K, class R>
__device__ __forceinline__ Mat2<R> ring_matrix(R r, R Ac, R m01) {
    const R hA = (R)0.5 * Ac;
    return {(R)1 + hA * r, m01, -hA * r * r * r, (R)1 - hA * r};
}
template <int K, class R>
__device__ __forceinline__ Mat2<R> ring_inverse(R r, R Ac, R m01) {
    const R hA = (R)0.5 * Ac;
    return {(R)1 - hA * r, -m01, hA * r * r * r, (R)1 + hA * r};
}
template <int K, class Op = OpMatLeft, class R>
__device__ __forceinline__ void ring_products(const R (&r)[K], const R (&Ac)[K], const R (&m01)[K], int np,
                                              Mat2<R>& Mf, Mat2<R>& Mb) {
    Mf = Mb = Op::template one<R>();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k < np) {
            if constexpr (Op::kDev) RingJump<R>(r[k], Ac[k], m01[k]).template multiply<false>(Mf);
            else Mf = OpMatLeft()(Mf, ring_matrix<K>(r[k], Ac[k], m01[k]));
        }
#pragma unroll
    for (int k = K - 1; k >= 0; --k)
        if (k < np) {
            if constexpr (Op::kDev) RingJump<R>(r[k], Ac[k], m01[k]).template multiply<true>(Mb);
            else Mb = OpMatLeft()(Mb, ring_inverse<K>(r[k], Ac[k], m01[k]));
        }
}

// a8 from the exclusive products Yf, Yb: B^(p) at this thread's rings and
// b_n; the regions' a, b to the tables where asked.  Takes an exchange and a
// barrier over the wake, after which the tables are complete.
template <class P, int K, class Op = OpMatLeft>
__device__ __forceinline__ void gm_region_solve(const WakeDev<P>& W, WakeCtas& C, GmShared<P>& s, int n, int p0,
                                                int np, const typename P::R (&r)[K], const typename P::R (&Ac)[K],
                                                const typename P::R (&m01)[K], const typename P::R (&Bc)[K],
                                                const typename P::R (&Cc)[K], const Mat2<typename P::R>& Yf,
                                                const Mat2<typename P::R>& Yb, bool tables, typename P::R (&bp)[K],
                                                typename P::R& bn) {
    using R = typename P::R;
    using A = typename P::A;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const A zeroA = acc_zero(A());
    // R walked to the end of the rings
    R Ra[K], Rb[K];
    {
        Mat2<R> Y = Op::whole(Yf);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (k < np) {
                if constexpr (Op::kDev) RingJump<R>(r[k], Ac[k], m01[k]).cross(Y.m00, Y.m10);
                else Y = OpMatLeft()(Y, ring_matrix<K>(r[k], Ac[k], m01[k]));
            }
            Ra[k] = Y.m00;
            Rb[k] = Y.m10;
        }
    }
    // R at the first region: its own product's, or as the thread before walked it
    const bool first = C.rank == 0 && tid == 0;
    R q0, q1;
    if constexpr (Op::kDev) {
        q0 = Op::whole(Yf).m00;
        q1 = Yf.m10;
    } else {
        q0 = shfl_up_t(Ra[K - 1], 1);
        q1 = shfl_up_t(Rb[K - 1], 1);
        if (lane == 31) {
            s.edge_r[0][warp] = Ra[K - 1];
            s.edge_r[1][warp] = Rb[K - 1];
        }
        if (C.size > 1 && tid == (int)blockDim.x - 1) {  // for the next block
            W.Ra[p0 + np] = Ra[K - 1];
            W.Rb[p0 + np] = Rb[K - 1];
        }
    }
    // ---- the Green's sums, D walked back
    A gl = zeroA, dl = zeroA;
    R gp[K], dp[K], Da[K], Db[K];
    {
        Mat2<R> Y = Op::whole(Yb);
#pragma unroll
        for (int k = K - 1; k >= 0; --k)
            if (k < np) {
                const R d0 = Y.m01, d1 = Y.m11;
                const R s0 = (R)0.25 * ((R)2 * Bc[k] + Ac[k] * Cc[k]);
                const R s1 = (R)0.25 * r[k] * ((R)4 * Cc[k] - (R)2 * Bc[k] * r[k] - Ac[k] * Cc[k] * r[k]);
                const R wr = Ra[k] * d1 - Rb[k] * d0;
                gp[k] = (s0 * d1 - s1 * d0) / wr;
                dp[k] = (Ra[k] * s1 - Rb[k] * s0) / wr;
                gl = acc_add_r(gl, gp[k]);
                dl = acc_add_r(dl, dp[k]);
                if constexpr (Op::kDev) RingJump<R>(r[k], Ac[k], m01[k]).cross_back(Y.m01, Y.m11);
                else Y = OpMatLeft()(Y, ring_inverse<K>(r[k], Ac[k], m01[k]));
                Da[k] = Y.m01;
                Db[k] = Y.m11;
            }
    }
    A g_tot, d_tot;
    Pair<A> gd = block_excl_scan_fwd_rev1(dl, gl, zeroA, s.g, d_tot, g_tot);
    if (C.size > 1) {
        const Pair<A>* buf = C.exchange(Pair<A>{d_tot, g_tot});
        A all;
        if (tid == 32 % (int)blockDim.x)
            gm_fold<true>(C, buf, zeroA, OpAdd(), [](Pair<A> v) { return v.y; }, s.pre_g.y, all);
        if (tid == 0)
            gm_fold<false>(C, buf, zeroA, OpAdd(), [](Pair<A> v) { return v.x; }, s.pre_g.x, s.tot_g.x);
        __syncthreads();
        gd.x = acc_add(s.pre_g.x, gd.x);
        gd.y = acc_add(s.pre_g.y, gd.y);
        d_tot = s.tot_g.x;
    }
    // ---- a8: the regions' a, b
    if constexpr (!Op::kDev) {
        if (lane == 0 && warp > 0) {
            q0 = s.edge_r[0][warp - 1];
            q1 = s.edge_r[1][warp - 1];
        }
        if (tid == 0 && C.rank > 0 && np > 0) {
            q0 = W.Ra[p0];
            q1 = W.Rb[p0];
        }
        if (first) {
            q0 = 1;
            q1 = 0;
        }
    }
    R ak[K], bk[K];
    {
        A Gs = gd.y;
#pragma unroll
        for (int k = K - 1; k >= 0; --k)
            if (k < np) {
                Gs = acc_add_r(Gs, gp[k]);
                const R G = acc_to_r(Gs);
                ak[k] = mul_rn(-G, k > 0 ? Ra[k - 1] : q0);
                bk[k] = mul_rn(-G, k > 0 ? Rb[k - 1] : q1);
            }
        A Hex = gd.x;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                const R H = acc_to_r(Hex);
                ak[k] += H * Da[k];
                bk[k] += H * Db[k];
                Hex = acc_add_r(Hex, dp[k]);
                if (tables) {
                    W.ak[p0 + k] = ak[k];
                    W.bk[p0 + k] = bk[k];
                }
            }
    }
    const R Hn = acc_to_r(d_tot);
    const R an = mul_rn(Hn, (R)0);  // region n: D_n = (0, 1)
    bn = mul_rn(Hn, (R)1);
    if (first && tables) {
        W.ak[n] = an;
        W.bk[n] = bn;
    }
    if (lane == 0) {
        s.edge_a[0][warp] = ak[0];
        s.edge_a[1][warp] = bk[0];
    }
    if (C.size > 1 && tid == 0 && np > 0 && !tables) {
        W.ak[p0] = ak[0];
        W.bk[p0] = bk[0];
    }
    R na = shfl_dn_t(ak[0], 1), nb = shfl_dn_t(bk[0], 1);
    C.sync();
    if (lane == 31) {
        if (tid + 1 < (int)blockDim.x) {
            na = s.edge_a[0][warp + 1];
            nb = s.edge_a[1][warp + 1];
        } else if (p0 + np < n) {
            na = W.ak[p0 + np];
            nb = W.bk[p0 + np];
        }
    }
    // B^(p) at the rings
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k < np) {
            const bool end = p0 + k + 1 == n;
            const R a1 = end ? an : k + 1 < K ? ak[k + 1 < K ? k + 1 : k] : na;
            const R b1 = end ? bn : k + 1 < K ? bk[k + 1 < K ? k + 1 : k] : nb;
            bp[k] = (R)0.5 * ((ak[k] + a1) * r[k] + (bk[k] + b1) / r[k]);
        }
}

// One evaluation of the fields (a4..a8) at the sorted rings of the wake: this
// thread's K radii (r, rlo), momenta u, logarithms and weights, and B^(b).
// `tables`: the region tables are written for the fields at other radii (they
// are complete after the caller's next barrier over the wake).
template <class P, int K, class Op = OpMatLeft>
struct GmFields {
    using R = typename P::R;
    using A = typename P::A;
    R psi[K], pb[K], g[K], dpr[K], dpz[K], bp[K];
    bool bad;

    __device__ __forceinline__ void evaluate(const WakeDev<P>& W, const Column<P>& col, WakeCtas& C, GmShared<P>& s,
                                             int n, int p0, int np, const R (&r)[K], const R (&rlo)[K],
                                             const R (&u)[K], const A (&lnr)[K], const A (&wa)[K],
                                             const A (&wha)[K], const R (&bb)[K], bool tables) {
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        const A zeroA = acc_zero(A());
        const Mat2<R> one = Op::template one<R>();
        // ---- a4
        Pair<A> loc = {zeroA, zeroA};
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                loc.x = acc_add(loc.x, wa[k]);
                loc.y = acc_add(loc.y, acc_mul_a(lnr[k], wa[k]));
            }
        Pair<A> tot;
        Pair<A> ex = block_excl_scan1<false>(loc, OpAddPair(), Pair<A>{zeroA, zeroA}, s.w, tot);
        if (C.size > 1) {
            const Pair<A>* buf = C.exchange(tot);
            if (tid == 0)
                gm_fold<false>(C, buf, Pair<A>{zeroA, zeroA}, OpAddPair(), [](Pair<A> v) { return v; }, s.pre_w,
                               s.tot_w);
            __syncthreads();
            ex = OpAddPair()(s.pre_w, ex);
            tot = s.tot_w;
        }
        const A Ltot = tot.y;

        // ---- a5, and the ring matrices of the B^(p) solve
        A S = ex.x, L = ex.y, tl = zeroA;
        R t[K], Ac[K], m01[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                const int p = p0 + k;
                const R w = acc_hi(wa[k]);
                const A X = make_radius(r[k], rlo[k]);
                const A Lsuf = acc_sub(Ltot, L);
                if (tables) {
                    W.regS[p] = S;
                    W.regL[p] = Lsuf;
                }
                const A r2 = acc_mul_a(X, X);
                const A Ir = r[k] < col.rmax ? acc_mul_r(r2, col.half_n) : col.Imax;
                const A psion = r[k] <= col.rmax ? acc_sub(col.c0, acc_mul_r(r2, col.quarter_n))
                                                 : acc_sub(zeroA, acc_mul_a(col.Imax, lnr[k]));
                psi[k] = acc_to_r(acc_add(acc_add(Lsuf, acc_mul_a(S, lnr[k])), psion));
                dpr[k] = acc_to_r(acc_div(acc_sub(acc_add(S, wha[k]), Ir), X));
                pb[k] = (R)1 + psi[k];
                g[k] = ((R)1 + u[k] * u[k] + pb[k] * pb[k]) / ((R)2 * pb[k]);
                t[k] = w * u[k] / (r[k] * pb[k]);
                S = acc_add(S, wa[k]);
                L = acc_add(L, acc_mul_a(lnr[k], wa[k]));
                tl = acc_add_r(tl, t[k]);
                Ac[k] = w / r[k] / pb[k];
                m01[k] = (R)0.5 * Ac[k] / r[k];
            }
        Mat2<R> Mf, Mb;
        ring_products<K, Op>(r, Ac, m01, np, Mf, Mb);
        A Ttot;
        Mat2<R> Yf, Yb, tf, tb;
        A Tex = block_excl_scan_sum_mats1<true, Op>(tl, Mf, Mb, zeroA, s.m, Yf, Yb, Ttot, tf, tb);
        if (C.size > 1) {
            const SumMats<A, R>* buf = C.exchange(SumMats<A, R>{Ttot, tf, tb});
            const int T = blockDim.x;
            Mat2<R> all;
            if (tid == 32 % T)
                gm_fold<true>(C, buf, one, Op(), [](SumMats<A, R> v) { return v.r; }, s.pre_r, all);
            if (tid == 64 % T)
                gm_fold<false>(C, buf, zeroA, OpAdd(), [](SumMats<A, R> v) { return v.t; }, s.pre_t, s.tot_t);
            if (tid == 0)
                gm_fold<false>(C, buf, one, Op(), [](SumMats<A, R> v) { return v.f; }, s.pre_f, all);
            __syncthreads();
            Tex = acc_add(s.pre_t, Tex);
            Ttot = s.tot_t;
            Yf = Op()(s.pre_f, Yf);
            Yb = Op()(s.pre_r, Yb);
        }

        // ---- a6 + a7
        R Bc[K], Cc[K];
        {
            A Tacc = Tex;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    const R w = acc_hi(wa[k]), wh = acc_hi(wha[k]);
                    if (tables) W.regT[p0 + k] = acc_to_r(acc_sub(Ttot, Tacc));
                    Tacc = acc_add_r(Tacc, t[k]);
                    const R above = acc_to_r(acc_sub(Ttot, Tacc));
                    dpz[k] = -(above + ((R)1 - wh / w) * t[k]);
                    ring_sources(w, r[k], u[k], pb[k], g[k], dpr[k], dpz[k], bb[k], Bc[k], Cc[k]);
                }
        }
        if (C.rank == 0 && tid == 0 && tables) {
            W.regS[n] = tot.x;
            W.regL[n] = zeroA;
            W.regT[n] = (R)0;
        }
        R bn;
        gm_region_solve<P, K, Op>(W, C, s, n, p0, np, r, Ac, m01, Bc, Cc, Yf, Yb, tables, bp, bn);
        // ---- guard
        bad = false;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np && (!(pb[k] > (R)0) || !real_finite(pb[k]) || !real_finite(dpr[k]) || !real_finite(dpz[k]) ||
                           !real_finite(bp[k]) || !real_finite(bb[k]) || !real_finite(g[k])))
                bad = true;
    }

    // the slice's ring dumps
    __device__ __forceinline__ void dump(const WakeDev<P>& W, int slice, int n, int np, const int (&id)[K],
                                         const R (&r)[K], const R (&u)[K], const R (&bb)[K]) const {
        if (!W.dump_r) return;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                const size_t row = (size_t)slice * n + id[k];
                W.dump_r[row] = r[k];
                if (W.dump_ur) {
                    W.dump_ur[row] = u[k];
                    W.dump_psi[row] = psi[k];
                    W.dump_dpr[row] = dpr[k];
                    W.dump_dpz[row] = dpz[k];
                    W.dump_bp[row] = bp[k];
                    W.dump_bb[row] = bb[k];
                }
            }
    }
};

// The order vote over the wake's rings (this thread's K radii r, np of them),
// with one more flag of the block's (OR over the blocks): true where every
// radius is in order.  edge: kGmWarps radii of shared memory, last: one.
template <int K, class R>
__device__ __forceinline__ bool gm_in_order(WakeCtas& C, const R (&r)[K], int n, int p0, int np, R* edge, R* last,
                                            bool& flag) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x;
    bool ok = true;
#pragma unroll
    for (int k = 1; k < K; ++k)
        if (k < np && r[k] < r[k - 1]) ok = false;
    R nxt = shfl_dn_t(r[0], 1);
    if (lane == 0) edge[warp] = r[0];
    if (np > 0 && (tid == T - 1 || p0 + np == n)) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k == np - 1) *last = r[k];
    }
    __syncthreads();
    if (lane == 31 && tid + 1 < T) nxt = edge[warp + 1];
    if (tid + 1 < T && np == K && p0 + K < n && nxt < r[K - 1]) ok = false;
    ok = __syncthreads_and(ok);
    if (C.size == 1) return ok;
    struct Edge {
        R first, last;
        int flags;
    };
    const Edge* v = C.exchange(Edge{edge[0], *last, (int)ok | (flag ? 2 : 0)});
    flag = false;
    Edge before = {};
    for (int i = 0; i < C.size; ++i) {
        const Edge b = C.slot(v, i);
        ok = ok && (b.flags & 1) != 0;
        flag = flag || (b.flags & 2) != 0;
        if (i > 0 && i * T * K < n && b.first < before.last) ok = false;
        before = b;
    }
    return ok;
}

// radii a[0, n) (16-byte aligned) into shared memory, loads in flight together
template <class R>
__device__ __forceinline__ void stage_radii(const R* a, int n, R* s) {
    constexpr int V = 16 / sizeof(R), U = 4;
    struct alignas(16) Vec {
        R v[V];
    };
    const int nv = n / V, T = blockDim.x;
    const Vec* av = reinterpret_cast<const Vec*>(a);
    for (int i0 = threadIdx.x; i0 < nv; i0 += U * T) {
        Vec x[U];
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (i0 + j * T < nv) x[j] = av[i0 + j * T];
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (i0 + j * T < nv) reinterpret_cast<Vec*>(s)[i0 + j * T] = x[j];
    }
    for (int i = nv * V + threadIdx.x; i < n; i += T) s[i] = a[i];
}

// psi, d_rho psi, d_zeta psi and B^(p) at a radius x >= 0 off the rings from
// the region tables (Eqs. b_theta_plasma..dpsi_dzeta); sR: the sorted radii
template <class P>
__device__ __forceinline__ void gm_fields_at(const WakeDev<P>& W, const Column<P>& col, const typename P::R* sR, int n,
                                             typename P::R x, typename P::R& psi, typename P::R& dpr,
                                             typename P::R& dpz, typename P::R& bp) {
    using R = typename P::R;
    using A = typename P::A;
    if (x > (R)0) {
        const int k = lower_bound_dev(sR, n, x);
        const A Sk = W.regS[k];
        psi = acc_to_r(acc_add(acc_add(W.regL[k], acc_mul_r(Sk, real_log(x))),
                               ion_psi(x, col.rmax, col.quarter_n, col.Imax, col.c0)));
        dpr = acc_to_r(acc_sub(Sk, ion_enclosed(x, col.rmax, col.half_n, col.Imax))) / x;
        dpz = -W.regT[k];
        bp = W.ak[k] * x + W.bk[k] / x;
    } else {
        psi = acc_to_r(acc_add(W.regL[0], ion_psi((R)0, col.rmax, col.quarter_n, col.Imax, col.c0)));
        dpr = 0;
        dpz = -W.regT[0];
        bp = 0;
    }
}

// The adaptive grids of one slice in this block's shared memory: extents and
// spacings per species, and B^(b) at the nodes.
constexpr int kGridNodesMax = 512;  // nodes of all species kept in shared memory
struct GridShared {
    double R[kMaxGridSpecies], dr[kMaxGridSpecies], inv_dr[kMaxGridSpecies];
    float Rf[kMaxGridSpecies];  // the smallest float not below R
    double BR[kMaxGridSpecies];  // B_N r_N
};
// ag_cell with a product in place of the quotient: the comparisons decide
__device__ __forceinline__ int grid_cell(double x, double dr, double inv_dr, int nr) {
    int j = (int)floor(x * inv_dr);
    if (j > nr - 1) j = nr - 1;
    if (j < 0) j = 0;
    while (j > 0 && (double)j * dr > x) --j;
    while (j < nr - 1 && (double)(j + 1) * dr <= x) ++j;
    return j;
}
__device__ __forceinline__ bool grid_beyond(const GridShared& G, int b, float rho) { return rho >= G.Rf[b]; }
__device__ __forceinline__ bool grid_beyond(const GridShared& G, int b, double rho) { return rho >= G.R[b]; }
// B^(b) at rho from the grids: linear between nodes inside, B_N r_N / rho beyond
template <class R>
__device__ __forceinline__ double grid_field(const GridShared& G, const R* B, int ns, int nr, R rho) {
    double v = 0.0;
    for (int b = 0; b < ns; ++b) {
        if (grid_beyond(G, b, rho)) {
            v += G.BR[b] / (double)rho;
        } else {
            const double x = (double)rho;
            const int j = grid_cell(x, G.dr[b], G.inv_dr[b], nr);
            const double t = (x - (double)j * G.dr[b]) / G.dr[b];
            const R* Bn = B + (size_t)b * (nr + 1);
            v += (1.0 - t) * (double)Bn[j] + t * (double)Bn[j + 1];
        }
    }
    return v;
}

// Shared memory of both marches: the radii of up to n_max rings, the ranks'
// scratch, and two slices' beam radii of up to kRegBeamCap each.
constexpr int kRegBeamCap = 2048;
template <class R>
__host__ __device__ inline int reg_sort_reals(int n) {  // a multiple of 16 bytes
    return (int)((RankSort<R>::bytes(n) + 15) / 16 * 16 / sizeof(R));
}
template <class R>
__host__ __device__ inline size_t reg_smem_bytes(int n_max, int beams) {
    return sizeof(R) * ((size_t)((n_max + 3) & ~3) + reg_sort_reals<R>(n_max) + (size_t)beams * kRegBeamCap);
}

// threads a block of the instantiation may have (the registers of 4 rings)
__host__ __device__ constexpr int reg_max_threads(int K) { return K > 2 ? 256 : 512; }

template <class P, int K>
__global__ void __launch_bounds__(reg_max_threads(K))
march_reg_kernel(const WakeDev<P>* __restrict__ wakes, const int32_t* __restrict__ order, int32_t max_slices,
                 int32_t mode) {
    using R = typename P::R;
    using A = typename P::A;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ctl[CTL_N];
    __shared__ int s_stop;
    __shared__ __align__(16) unsigned char s_part[2 * kPartBuf];
    __shared__ GmShared<P> s_ev;
    __shared__ R s_edge[kGmWarps], s_last;
    __shared__ typename RankSort<R>::KT s_keys[64];
    __shared__ GridShared s_grid;
    __shared__ R s_nodes[kGridNodesMax];

    const uint64_t t_launch = global_ns();
    WakeCtas C;
    {
        unsigned r, c;
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(c));
        C.rank = (int)r;
        C.size = (int)c;
        C.part = s_part;
    }
    C.start();
    const int wi = blockIdx.x / C.size;
    const WakeDev<P>& W = wakes[order ? order[wi] : wi];
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gt = C.rank * T + tid, GT = C.size * T;
    const int n = W.n;
    const int p0 = min(n, gt * K), np = min(K, n - p0);
    const bool lead = C.rank == 0 && tid == 0;

    R* sR = reinterpret_cast<R*>(smem);  // all radii (staged when searched)
    const int n4 = (n + 3) & ~3;
    RankSort<R> sorter(sR, n, sR + n4);
    R* sB = sR + n4 + reg_sort_reals<R>(n);  // the slice's beam radii

    if (tid < CTL_N) s_ctl[tid] = W.ctl[tid];
    __syncthreads();
    if (s_ctl[CTL_STATUS] != 0) return;
    int slice = s_ctl[CTL_NEXT];
    int buf = s_ctl[CTL_BUF];
    int has_prev = s_ctl[CTL_PREV];
    int status = 0, fail = -1;
    const bool query = mode != MODE_MARCH;
    const int s_end = query ? slice + 1 : min(W.n_steps, slice + max_slices);
    const Column<P> col(W);
    const R dxi = (R)W.dxi;
    const R inv_2pi_dxi = (R)(1.0 / (6.283185307179586476925286766559 * W.dxi));

    // the grids: extents once per launch; nodes in shared memory where they fit
    const int nr = W.grid_nr, ns = W.n_species, nn = ns * (nr + 1);
    R* nodes = nr > 0 && nn > kGridNodesMax ? W.agB : s_nodes;
    const bool shared_nodes = nodes == s_nodes;
    if (nr > 0) {
        if (tid < ns) {
            const double Rb = ag_extent(W, tid);
            s_grid.R[tid] = Rb;
            s_grid.dr[tid] = Rb / nr;
            s_grid.inv_dr[tid] = nr / Rb;
            s_grid.Rf[tid] = __double2float_ru(Rb);
        }
        if (C.rank == 0)  // (ordered by the order vote's barrier)
            for (int i = tid; i < nn; i += T) W.agB[i] = 0;
        __syncthreads();
    }

    R r[K], rlo[K], u[K], fr[K], fu[K];
    int id[K];
    A wa[K], wha[K];
    auto load = [&]() {
        load_rings<K>(W.rho[buf], p0, np, r, (R)1);
        load_rings<K>(W.rho_lo, p0, np, rlo, (R)0);
        load_rings<K>(W.ur[buf], p0, np, u, (R)0);
        load_rings<K>(W.frho[buf], p0, np, fr, (R)0);
        load_rings<K>(W.fur[buf], p0, np, fu, (R)0);
        load_rings<K>(W.rid[buf], p0, np, id, 0);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) ring_weights(W.ctab, W.w, W.wh, id[k], wa[k], wha[k]);
    };
    auto store = [&](int b, int k, int p) {
        W.rho[b][p] = r[k];
        W.ur[b][p] = u[k];
        W.frho[b][p] = fr[k];
        W.fur[b][p] = fu[k];
        W.rid[b][p] = id[k];
    };
    load();
    // (every thread's low parts are read: they have one buffer)
    C.sync();

    const int slice0 = slice;
    uint64_t t_start = 0;
    for (; slice < s_end; ++slice) {
        // time budget (thread 0 decides, read after the order check's barrier)
        if (W.budget_ns > 0 && tid == 0) {
            const uint64_t now = global_ns();
            if (slice == slice0) t_start = now;
            s_stop = slice > slice0 && now - t_start >= (uint64_t)W.budget_ns;
        }
        // this slice's beam (the loads overlap the order vote)
        const bool have_beam = W.nb > 0 && slice < W.n_steps;
        int b0 = 0, m = 0;
        R qtot = 0;
        if (have_beam) {
            b0 = W.boff[slice];
            m = W.boff[slice + 1] - b0;
            qtot = W.bTot[slice];
        }
        // ---------------- a2: order vote; rings that crossed move to their ranks (stable)
        if (W.budget_ns > 0) __syncthreads();
        bool stop = W.budget_ns > 0 && s_stop;
        const bool in_order = gm_in_order<K>(C, r, n, p0, np, s_edge, &s_last, stop);
        if (stop) break;
        if (!in_order) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];
            C.sync();
            stage_radii(W.rho[buf], n, sR);
            __syncthreads();
            sorter.prepare(s_keys);
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    const int p = sorter.place(p0 + k, r[k]);
                    store(buf ^ 1, k, p);
                    W.rho_lo[p] = rlo[k];
                }
            buf ^= 1;
            C.sync();
            load();
        }
        // the radii and the region tables serve other radii than the rings'
        const bool tables = query || m > 0;
        if (tables && in_order) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];  // (read after the scans' barriers)
        }
        const bool staged = m <= kRegBeamCap;
        if (m > 0 && staged && (nr == 0 || query)) {
            for (int q = tid; q < m; q += T) sB[q] = W.br[b0 + q];
            __syncthreads();
        }
        const R* beamR = staged ? sB : (W.br + b0);

        // ---------------- adaptive grids: B^(b) at the nodes of this slice
        if (nr > 0) {
            for (int q = gt; q < m; q += GT) {  // each particle's charge reaches the nodes above it
                const int64_t k = W.bidx[b0 + q];
                const int b = ag_species(W, k);
                const int j = grid_cell(W.rc[k], s_grid.dr[b], s_grid.inv_dr[b], nr) + 1;
                atomicAdd(W.agB + (size_t)b * (nr + 1) + j, (R)W.qw[k]);
            }
            C.sync();
            // a warp per species: the running charge over the nodes (every
            // block for itself; block 0 for all where the nodes stay global)
            if ((shared_nodes || C.rank == 0) && warp < min(ns, T / 32)) {
                for (int b = warp; b < ns; b += T / 32) {
                    const R* Q = W.agB + (size_t)b * (nr + 1);
                    R* B = nodes + (size_t)b * (nr + 1);
                    const double dr = s_grid.dr[b];
                    double carry = 0.0;
                    for (int base = 1; base <= nr; base += 32) {
                        const int j = base + lane;
                        const double v = j <= nr ? (double)Q[j] : 0.0;
                        const double in = carry + warp_incl_scan<false>(v, OpAdd());
                        carry = shfl_idx_t(in, 31);
                        if (j <= nr) {
                            const R Bj = (R)(in / (6.283185307179586476925286766559 * W.dxi * ((double)j * dr)));
                            B[j] = Bj;
                            if (j == nr) s_grid.BR[b] = (double)Bj * s_grid.R[b];
                        }
                    }
                    if (lane == 0) B[0] = 0;
                }
            }
            if (shared_nodes) {
                __syncthreads();
            } else {
                C.sync();
                if (tid < ns) s_grid.BR[tid] = (double)nodes[(size_t)tid * (nr + 1) + nr] * s_grid.R[tid];
                __syncthreads();
            }
        }

        // ---------------- a3: beam field at the rings
        R bb[K];
        A lnr[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            bb[k] = 0;
            lnr[k] = acc_zero(A());
            if (k < np) {
                if (nr > 0) {
                    bb[k] = (R)grid_field(s_grid, nodes, ns, nr, r[k]);
                } else if (m > 0 && r[k] > (R)0) {
                    const int lb = lower_bound_dev(beamR, m, r[k]);
                    const R Q = lb < m ? W.bE[b0 + lb] : qtot;
                    bb[k] = Q * inv_2pi_dxi / r[k];
                }
                lnr[k] = ring_log(W.ctab, id[k], r[k], rlo[k]);
            }
        }
        // ---------------- a4..a8
        // (matrices less the identity where their rounding shows: see ring_jump.cuh)
        using Op = typename std::conditional<K >= 3 && std::is_same<P, PrecMixed>::value, OpMatDevLeft, OpMatLeft>::type;
        GmFields<P, K, Op> F;
        F.evaluate(W, col, C, s_ev, n, p0, np, r, rlo, u, lnr, wa, wha, bb, tables);
        if (tables) stage_radii(W.rho[buf], n, sR);
        if (!query) F.dump(W, slice, n, np, id, r, u, bb);
        const bool bad = wake_vote(C, F.bad, false);

        if (nr > 0 && !query && m > 0) {
            // ---------------- adaptive grids: the plasma fields at the nodes
            for (int i = gt; i < nn; i += GT) {
                const int b = i / (nr + 1), j = i - b * (nr + 1);
                const R x = (R)((double)j * s_grid.dr[b]);
                R psi, dprv, dpz, bpv;
                gm_fields_at(W, col, sR, n, x, psi, dprv, dpz, bpv);
                if (x > (R)0) bpv = bpv + (R)grid_field(s_grid, nodes, ns, nr, x);
                R* F4 = W.agF + (size_t)i * 4;
                F4[0] = psi;
                F4[1] = dprv;
                F4[2] = dpz;
                F4[3] = bpv;
            }
            C.sync();
            for (int q = gt; q < m; q += GT) {
                const int64_t kc = W.bidx[b0 + q];
                const int b = ag_species(W, kc);
                const double dr = s_grid.dr[b];
                const double x = W.rc[kc];  // the caller's FP64 radius: node membership as the oracle's
                const int j = grid_cell(x, dr, s_grid.inv_dr[b], nr);
                const R t = (R)((x - (double)j * dr) / dr);
                const R* F0 = W.agF + ((size_t)b * (nr + 1) + j) * 4;
                const R* F1 = F0 + 4;
                const int64_t o = b0 + q;
                W.out_ez[o] = -(((R)1 - t) * F0[2] + t * F1[2]);
                W.out_wr[o] = -(((R)1 - t) * F0[1] + t * F1[1]);
                W.out_bt[o] = ((R)1 - t) * F0[3] + t * F1[3];
                W.out_psi[o] = ((R)1 - t) * F0[0] + t * F1[0];
            }
        }
        // (the nodes' last use of this slice is behind a barrier: the node
        // fields' or the vote's; the next deposits come after the order vote)
        if (nr > 0 && C.rank == 0)
            for (int i = tid; i < nn; i += T) W.agB[i] = 0;

        // ---------------- a9: fields on beam particles (or query radii)
        if (query || (nr == 0 && m > 0)) {
            const int64_t nq = query ? W.nq : (int64_t)m;
            for (int64_t q = gt; q < nq; q += GT) {
                R x;
                if (query) x = (R)W.rq[q];
                else x = staged ? beamR[q] : W.br[b0 + q];
                R psi, dprv, dpz, bpv, bbv = 0;
                gm_fields_at(W, col, sR, n, x, psi, dprv, dpz, bpv);
                if (x > (R)0) {
                    if (!query) {
                        bbv = W.bQs[b0 + q] * inv_2pi_dxi / x;
                    } else if (m > 0) {
                        const int lb = lower_bound_dev(W.br + b0, m, x);
                        const R Q = lb < m ? W.bE[b0 + lb] : qtot;
                        bbv = Q * inv_2pi_dxi / x;
                    }
                }
                if (!query) {
                    const int64_t o = b0 + q;
                    W.out_ez[o] = -dpz;
                    W.out_wr[o] = -dprv;
                    W.out_bt[o] = bpv + bbv;
                    W.out_psi[o] = psi;
                } else {
                    if (W.q_ez) W.q_ez[q] = -dpz;
                    if (W.q_wr) W.q_wr[q] = -dprv;
                    if (W.q_bt) W.q_bt[q] = bpv + bbv;
                    if (W.q_psi) W.q_psi[q] = psi;
                }
            }
        }
        if (query) break;
        if (bad) {
            status = 4;
            fail = slice;
            ++slice;
            break;
        }

        // ---------------- a10: AB2 push to the next slice
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                R gr = u[k] / F.pb[k];
                R gu = F.g[k] * F.dpr[k] / F.pb[k] - (F.bp[k] + bb[k]);
                R rn = r[k], rl = rlo[k], un;
                if (has_prev) {
                    radius_add(rn, rl, dxi * ((R)1.5 * gr - (R)0.5 * fr[k]));
                    un = u[k] + dxi * ((R)1.5 * gu - (R)0.5 * fu[k]);
                } else {
                    radius_add(rn, rl, dxi * gr);
                    un = u[k] + dxi * gu;
                }
                if (rn < (R)0) {
                    rn = -rn;
                    rl = -rl;
                    un = -un;
                    gr = -gr;
                    gu = -gu;
                }
                r[k] = rn;
                rlo[k] = rl;
                u[k] = un;
                fr[k] = gr;
                fu[k] = gu;
            }
        has_prev = 1;
    }
    C.sync();  // (every read of the tables and radii is done)
    if (!query) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                store(buf, k, p0 + k);
                W.rho_lo[p0 + k] = rlo[k];
            }
    }
    if (lead) {
        if (!query) put_march_times(W.ctl, t_launch);
        W.ctl[CTL_NEXT] = query ? s_ctl[CTL_NEXT] : slice;
        W.ctl[CTL_BUF] = buf;
        W.ctl[CTL_PREV] = has_prev;
        if (status) {
            W.ctl[CTL_STATUS] = status;
            W.ctl[CTL_FAIL] = fail;
        }
    }
}

// the beam source of a stage: w1 x (slice a) + w2 x (slice b, if m2 > 0)
template <class R>
struct StageSource {
    const R *r1, *r2;  // the slices' sorted radii (staged, or global)
    int b1, m1, b2, m2;
    R w1, w2, q1, q2;
};
template <class P>
__device__ __forceinline__ typename P::R stage_beam_field(const WakeDev<P>& W, const StageSource<typename P::R>& S,
                                                          typename P::R r, typename P::R inv_2pi_dxi) {
    using R = typename P::R;
    if (!(r > (R)0)) return (R)0;
    R bb = 0;
    if (S.m1 > 0) {
        const int lb = lower_bound_dev(S.r1, S.m1, r);
        bb += S.w1 * (lb < S.m1 ? W.bE[S.b1 + lb] : S.q1);
    }
    if (S.m2 > 0) {
        const int lb = lower_bound_dev(S.r2, S.m2, r);
        bb += S.w2 * (lb < S.m2 ? W.bE[S.b2 + lb] : S.q2);
    }
    return bb * inv_2pi_dxi / r;
}

// The RK4 march (the stages of march_rk4.cuh).  The state and the weighted
// derivative sums stay with the thread of the ring's place at the slice's
// start; a stage whose state is out of that order is carried to the threads
// of its own order through the wake's stage arrays and its derivatives back.
// The guard is voted once per slice: a stage after a failed one computes on
// what there is and the slice's update is dropped.
template <class P, int K>
__global__ void __launch_bounds__(reg_max_threads(K))
march_rk4_reg_kernel(const WakeDev<P>* __restrict__ wakes, const int32_t* __restrict__ order, int32_t max_slices,
                     int32_t mode) {
    using R = typename P::R;
    using A = typename P::A;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ctl[CTL_N];
    __shared__ int s_stop;
    __shared__ __align__(16) unsigned char s_part[2 * kPartBuf];
    __shared__ GmShared<P> s_ev;
    __shared__ R s_edge[kGmWarps], s_last;
    __shared__ typename RankSort<R>::KT s_keys[64];

    const uint64_t t_launch = global_ns();
    WakeCtas C;
    {
        unsigned r, c;
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
        asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(c));
        C.rank = (int)r;
        C.size = (int)c;
        C.part = s_part;
    }
    C.start();
    const int wi = blockIdx.x / C.size;
    const WakeDev<P>& W = wakes[order ? order[wi] : wi];
    const int T = blockDim.x, tid = threadIdx.x;
    const int gt = C.rank * T + tid, GT = C.size * T;
    const int n = W.n;
    const int p0 = min(n, gt * K), np = min(K, n - p0);
    const bool lead = C.rank == 0 && tid == 0;

    R* sR = reinterpret_cast<R*>(smem);
    const int n4 = (n + 3) & ~3;
    RankSort<R> sorter(sR, n, sR + n4);
    R* sB = sR + n4 + reg_sort_reals<R>(n);  // beam radii of this slice and the next
    R* sB2 = sB + kRegBeamCap;

    if (tid < CTL_N) s_ctl[tid] = W.ctl[tid];
    __syncthreads();
    if (s_ctl[CTL_STATUS] != 0) return;
    int slice = s_ctl[CTL_NEXT];
    int buf = s_ctl[CTL_BUF];
    int status = 0, fail = -1;
    const bool query = mode != MODE_MARCH;
    const int s_end = query ? slice + 1 : min(W.n_steps, slice + max_slices);
    const Column<P> col(W);
    const R dxi = (R)W.dxi;
    const R inv_2pi_dxi = (R)(1.0 / (6.283185307179586476925286766559 * W.dxi));

    R r[K], rlo[K], u[K], kr[K], ku[K], sum_r[K], sum_u[K];
    int id[K];
    A wa[K], wha[K];
    auto load = [&]() {
        load_rings<K>(W.rho[buf], p0, np, r, (R)1);
        load_rings<K>(W.rho_lo, p0, np, rlo, (R)0);
        load_rings<K>(W.ur[buf], p0, np, u, (R)0);
        load_rings<K>(W.rid[buf], p0, np, id, 0);
    };
    auto weights = [&](const int (&ids)[K]) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) ring_weights(W.ctab, W.w, W.wh, ids[k], wa[k], wha[k]);
    };
    load();
    C.sync();  // (every thread's low parts are read: they have one buffer)

    // the radii of every thread's rings (base[p] written by the caller), their ranks prepared
    auto rank = [&](const R* base) {
        C.sync();
        stage_radii(base, n, sR);
        __syncthreads();
        sorter.prepare(s_keys);
    };

    const int slice0 = slice;
    uint64_t t_start = 0;
    bool summed = false;
    for (; slice < s_end; ++slice) {
        // time budget (thread 0 decides, read after the order check's barrier)
        if (W.budget_ns > 0 && tid == 0) {
            const uint64_t now = global_ns();
            if (slice == slice0) t_start = now;
            s_stop = slice > slice0 && now - t_start >= (uint64_t)W.budget_ns;
        }
        // ---------------- the slice's beam and the next slice's (the loads overlap the order vote)
        const bool have_beam = W.nb > 0 && slice < W.n_steps;
        int b0 = 0, m = 0, b1 = 0, m1 = 0;
        R qtot = 0, qtot1 = 0;
        if (have_beam) {
            b0 = W.boff[slice];
            m = W.boff[slice + 1] - b0;
            qtot = W.bTot[slice];
            if (slice + 1 < W.n_steps) {
                b1 = W.boff[slice + 1];
                m1 = W.boff[slice + 2] - b1;
                qtot1 = W.bTot[slice + 1];
            }
        }
        // ---------------- a2: order vote; rings that crossed move to their ranks (stable)
        if (W.budget_ns > 0) __syncthreads();
        bool stop = W.budget_ns > 0 && s_stop;
        const bool in_order = gm_in_order<K>(C, r, n, p0, np, s_edge, &s_last, stop);
        if (stop) break;
        if (!in_order) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];
            rank(W.rho[buf]);
            const int nb = buf ^ 1;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    const int p = sorter.place(p0 + k, r[k]);
                    W.rho[nb][p] = r[k];
                    W.rho_lo[p] = rlo[k];
                    W.ur[nb][p] = u[k];
                    W.rid[nb][p] = id[k];
                }
            buf = nb;
            C.sync();
            load();
        }
        const bool tables = query || m > 0;
        if (tables && in_order) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];  // (read after the scans' barriers)
        }
        const bool staged = m <= kRegBeamCap, staged1 = m1 <= kRegBeamCap;
        if (staged)
            for (int q = tid; q < m; q += T) sB[q] = W.br[b0 + q];
        if (staged1)
            for (int q = tid; q < m1; q += T) sB2[q] = W.br[b1 + q];
        __syncthreads();
        const R* beamR = staged ? sB : W.br + b0;
        const R* beamR1 = staged1 ? sB2 : W.br + b1;

        // ---------------- stage 1 at (xi_n, y_n): the slice's fields
        GmFields<P, K> F;
        R bb[K];
        A lnr[K];
        auto source = [&](const StageSource<R>& S, const R (&x)[K], const R (&xlo)[K], const int (&ids)[K]) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                bb[k] = 0;
                lnr[k] = acc_zero(A());
                if (k < np) {
                    bb[k] = stage_beam_field(W, S, x[k], inv_2pi_dxi);
                    lnr[k] = ring_log(W.ctab, ids[k], x[k], xlo[k]);
                }
            }
        };
        weights(id);
        source(StageSource<R>{beamR, beamR1, b0, m, 0, 0, (R)1, (R)0, qtot, (R)0}, r, rlo, id);
        F.evaluate(W, col, C, s_ev, n, p0, np, r, rlo, u, lnr, wa, wha, bb, tables);
        bool bad = F.bad;
        if (!query) F.dump(W, slice, n, np, id, r, u, bb);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                kr[k] = u[k] / F.pb[k];
                ku[k] = F.g[k] * F.dpr[k] / F.pb[k] - (F.bp[k] + bb[k]);
                sum_r[k] = kr[k];
                sum_u[k] = ku[k];
            }
        summed = true;

        // ---------------- a9: fields on beam particles (or query radii)
        if (tables) {
            stage_radii(W.rho[buf], n, sR);
            __syncthreads();
            const int64_t nq = query ? W.nq : (int64_t)m;
            for (int64_t q = gt; q < nq; q += GT) {
                R x;
                if (query) x = (R)W.rq[q];
                else x = staged ? beamR[q] : W.br[b0 + q];
                R psi, dprv, dpz, bpv, bbv = 0;
                if (x > (R)0) {
                    const int k = lower_bound_dev(sR, n, x);
                    const A Sk = W.regS[k];
                    const R lnx = real_log(x);
                    const A x2 = acc_sq(x);
                    const A psion = x <= col.rmax ? acc_sub(col.c0, acc_mul_r(x2, col.quarter_n))
                                                  : acc_sub(acc_zero(A()), acc_mul_r(col.Imax, lnx));
                    const A Ix = x < col.rmax ? acc_mul_r(x2, col.half_n) : col.Imax;
                    psi = acc_to_r(acc_add(acc_add(W.regL[k], acc_mul_r(Sk, lnx)), psion));
                    dprv = acc_to_r(acc_sub(Sk, Ix)) / x;
                    dpz = -W.regT[k];
                    bpv = W.ak[k] * x + W.bk[k] / x;
                    if (!query) {
                        bbv = W.bQs[b0 + q] * inv_2pi_dxi / x;
                    } else if (m > 0) {
                        const int lb = lower_bound_dev(beamR, m, x);
                        const R Q = lb < m ? W.bE[b0 + lb] : qtot;
                        bbv = Q * inv_2pi_dxi / x;
                    }
                } else {
                    psi = acc_to_r(acc_add(W.regL[0], col.c0));
                    dprv = 0;
                    dpz = -W.regT[0];
                    bpv = 0;
                }
                if (!query) {
                    const int64_t o = b0 + q;
                    W.out_ez[o] = -dpz;
                    W.out_wr[o] = -dprv;
                    W.out_bt[o] = bpv + bbv;
                    W.out_psi[o] = psi;
                } else {
                    if (W.q_ez) W.q_ez[q] = -dpz;
                    if (W.q_wr) W.q_wr[q] = -dprv;
                    if (W.q_bt) W.q_bt[q] = bpv + bbv;
                    if (W.q_psi) W.q_psi[q] = psi;
                }
            }
        }
        if (query) break;

        // ---------------- stages 2-4
#pragma unroll 1
        for (int stg = 0; stg < 3; ++stg) {
            const R cst = stg < 2 ? (R)0.5 : (R)1, wst = stg < 2 ? (R)2 : (R)1;
            // the stage state, mirrored at the axis
            R sr[K], sl[K], su[K], sg[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                sr[k] = (R)1;
                sl[k] = su[k] = (R)0;
                sg[k] = (R)1;
                if (k < np) {
                    R x = r[k], xl = rlo[k];
                    radius_add(x, xl, cst * dxi * kr[k]);
                    const R v = u[k] + cst * dxi * ku[k];
                    sg[k] = x < (R)0 ? (R)-1 : (R)1;
                    sr[k] = sg[k] * x;
                    sl[k] = sg[k] * xl;
                    su[k] = sg[k] * v;
                }
            }
            bool none = false;
            const bool same = gm_in_order<K>(C, sr, n, p0, np, s_edge, &s_last, none);
            int ids[K], at[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                ids[k] = id[k];
                at[k] = p0 + k;
            }
            if (!same) {
                R* base = W.rho[buf ^ 1];
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < np) base[p0 + k] = sr[k];
                rank(base);
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < np) {
                        const int p = sorter.place(p0 + k, sr[k]);
                        W.rk_r[p] = sr[k];
                        W.rk_rlo[p] = sl[k];
                        W.rk_u[p] = su[k];
                        W.rk_sg[p] = sg[k];
                        W.rid[buf ^ 1][p] = id[k];
                        W.rk_perm[p] = p0 + k;
                    }
                C.sync();
                load_rings<K>(W.rk_r, p0, np, sr, (R)1);
                load_rings<K>(W.rk_rlo, p0, np, sl, (R)0);
                load_rings<K>(W.rk_u, p0, np, su, (R)0);
                load_rings<K>(W.rk_sg, p0, np, sg, (R)1);
                load_rings<K>(W.rid[buf ^ 1], p0, np, ids, 0);
                load_rings<K>(W.rk_perm, p0, np, at, 0);
            }
            weights(ids);
            if (stg < 2)
                source(StageSource<R>{beamR, beamR1, b0, m, b1, m1, (R)0.5, (R)0.5, qtot, qtot1}, sr, sl, ids);
            else
                source(StageSource<R>{beamR1, beamR1, b1, m1, 0, 0, (R)1, (R)0, qtot1, (R)0}, sr, sl, ids);
            F.evaluate(W, col, C, s_ev, n, p0, np, sr, sl, su, lnr, wa, wha, bb, false);
            bad = bad || F.bad;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    kr[k] = sg[k] * (su[k] / F.pb[k]);
                    ku[k] = sg[k] * (F.g[k] * F.dpr[k] / F.pb[k] - (F.bp[k] + bb[k]));
                }
            if (!same) {  // back to the threads of the slice's order
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < np) {
                        W.rk_kr[at[k]] = kr[k];
                        W.rk_ku[at[k]] = ku[k];
                    }
                C.sync();
                load_rings<K>(W.rk_kr, p0, np, kr, (R)0);
                load_rings<K>(W.rk_ku, p0, np, ku, (R)0);
            }
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    sum_r[k] += wst * kr[k];
                    sum_u[k] += wst * ku[k];
                }
        }
        if (wake_vote(C, bad, false)) {
            status = 4;
            fail = slice;
            ++slice;
            break;
        }

        // ---------------- y_{n+1} = y_n + h/6 (k1 + 2 k2 + 2 k3 + k4), reflection
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                R x = r[k], xl = rlo[k];
                radius_add(x, xl, dxi / (R)6 * sum_r[k]);
                R v = u[k] + dxi / (R)6 * sum_u[k];
                if (x < (R)0) {
                    x = -x;
                    xl = -xl;
                    v = -v;
                }
                r[k] = x;
                rlo[k] = xl;
                u[k] = v;
            }
    }
    C.sync();  // (every read of the tables and radii is done)
    // (the derivative sums are left where the march of march_rk4.cuh keeps them)
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k < np) {
            const int p = p0 + k;
            if (summed) {
                W.frho[0][p] = sum_r[k];
                W.fur[0][p] = sum_u[k];
            }
            if (!query) {
                W.rho[buf][p] = r[k];
                W.rho_lo[p] = rlo[k];
                W.ur[buf][p] = u[k];
                W.rid[buf][p] = id[k];
            }
        }
    if (lead) {
        if (!query) put_march_times(W.ctl, t_launch);
        W.ctl[CTL_NEXT] = query ? s_ctl[CTL_NEXT] : slice;
        W.ctl[CTL_BUF] = buf;
        W.ctl[CTL_PREV] = 0;
        if (status) {
            W.ctl[CTL_STATUS] = status;
            W.ctl[CTL_FAIL] = fail;
        }
    }
}

}  // namespace gbwake
