// march_reg_ions.cuh -- the two-species march of march_ions.cuh with the
// rings in registers (see march_reg.cuh), for shapes of up to 2 rings of each
// species per thread.
//
// Besides what march_reg.cuh says of the global-memory marches, the
// two-species one searched the other species' radii three times per ring (for
// psi and d_rho psi, for d_zeta psi, for B^(p) at the ions); here a ring
// keeps the place and weights it found first.  The own-species fields and
// B^(p) at the electron rings, which the other species gathers from any
// block, stay in global memory.  The electrons' solve matrices depend on psi
// only and travel with both species' t sums: nine barriers over the wake per
// slice (the order vote, the two species' scans, own fields, t and matrices,
// own d_zeta psi, Green's sums, regions, B^(p), the guard).
// Measured on GB300, 24 wakes of 500-4000 cells in one batch: 62 -> 47 us
// per slice (FP64, 8 wakes: 276 -> 233, its FP64 pipe's).
#pragma once

#include "march_reg.cuh"

namespace gbwake {

template <class P, int K>
__global__ void __launch_bounds__(512)
march_ions_reg_kernel(const WakeDev<P>* __restrict__ wakes, const int32_t* __restrict__ order, int32_t max_slices,
                      int32_t mode) {
    using R = typename P::R;
    using A = typename P::A;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ctl[CTL_N];
    __shared__ int s_stop;
    __shared__ __align__(16) unsigned char s_part[2 * kPartBuf];
    __shared__ GmShared<P> s_ev;
    __shared__ Pair<A> s_w1[kGmWarps], s_fold[4];
    __shared__ A s_t1[kGmWarps], s_tf[4];
    __shared__ R s_edge[2][kGmWarps], s_last[2];
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
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gt = C.rank * T + tid, GT = C.size * T;
    const int n = W.n, N = W.n_ion;
    const int q0 = min(N, gt * K), np = min(K, N - q0);  // this thread's rings of each species
    const bool lead = C.rank == 0 && tid == 0;
    const R qm[2] = {(R)-1, (R)W.ion_qm};

    R* sR = reinterpret_cast<R*>(smem);  // both segments' radii
    const int n4 = (n + 3) & ~3;
    R* s_sort = sR + n4;
    R* sB = s_sort + reg_sort_reals<R>(n);

    if (tid < CTL_N) s_ctl[tid] = W.ctl[tid];
    __syncthreads();
    if (s_ctl[CTL_STATUS] != 0) return;
    int slice = s_ctl[CTL_NEXT];
    int buf = s_ctl[CTL_BUF];
    int has_prev = s_ctl[CTL_PREV];
    int status = 0, fail = -1;
    const bool query = mode != MODE_MARCH;
    const int s_end = query ? slice + 1 : min(W.n_steps, slice + max_slices);

    const R edge = (R)W.rho_max;
    const A Xe = acc_from_d(W.rho_max, A());
    const A ln_e = acc_from_d(log(W.rho_max), A());
    const A inv_e = acc_from_d(1.0 / W.rho_max, A());
    const R dxi = (R)W.dxi;
    const R inv_2pi_dxi = (R)(1.0 / (6.283185307179586476925286766559 * W.dxi));
    const A zeroA = acc_zero(A());
    const Pair<A> zeroP = {zeroA, zeroA};

    R r[2][K], rlo[2][K], u[2][K], fr[2][K], fu[2][K], c[2][K], ch[2][K];
    int id[2][K];
    auto load = [&]() {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int p0 = s * N + q0;
            load_rings<K>(W.rho[buf], p0, np, r[s], (R)1);
            load_rings<K>(W.rho_lo, p0, np, rlo[s], (R)0);
            load_rings<K>(W.ur[buf], p0, np, u[s], (R)0);
            load_rings<K>(W.frho[buf], p0, np, fr[s], (R)0);
            load_rings<K>(W.fur[buf], p0, np, fu[s], (R)0);
            load_rings<K>(W.rid[buf], p0, np, id[s], 0);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                c[s][k] = k < np ? W.w[id[s][k]] : (R)0;
                ch[s][k] = k < np ? W.wh[id[s][k]] : (R)0;
            }
    };
    auto store = [&](int b, int s, int k, int p) {
        W.rho[b][p] = r[s][k];
        W.ur[b][p] = u[s][k];
        W.frho[b][p] = fr[s][k];
        W.fur[b][p] = fu[s][k];
        W.rid[b][p] = id[s][k];
    };
    load();
    C.sync();  // (every thread's low parts are read: they have one buffer)

    const int slice0 = slice;
    uint64_t t_start = 0;
    for (; slice < s_end; ++slice) {
        // time budget (thread 0 decides, read after the order check's barrier)
        if (W.budget_ns > 0 && tid == 0) {
            const uint64_t now = global_ns();
            if (slice == slice0) t_start = now;
            s_stop = slice > slice0 && now - t_start >= (uint64_t)W.budget_ns;
        }
        // the slice's beam (the loads overlap the order vote); the radii, for
        // the searches of every block
        const bool have_beam = W.nb > 0 && slice < W.n_steps;
        int b0 = 0, m = 0;
        R qtot = 0;
        if (have_beam) {
            b0 = W.boff[slice];
            m = W.boff[slice + 1] - b0;
            qtot = W.bTot[slice];
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][s * N + q0 + k] = r[s][k];
        // ---------------- a2: order vote; rings that crossed move to their ranks (stable)
        if (W.budget_ns > 0) __syncthreads();
        bool stop = W.budget_ns > 0 && s_stop;
        bool ok = true;
        R nxt[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
#pragma unroll
            for (int k = 1; k < K; ++k)
                if (k < np && r[s][k] < r[s][k - 1]) ok = false;
            nxt[s] = shfl_dn_t(r[s][0], 1);
            if (lane == 0) s_edge[s][warp] = r[s][0];
            if (np > 0 && (tid == T - 1 || q0 + np == N)) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k == np - 1) s_last[s] = r[s][k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (lane == 31 && tid + 1 < T) nxt[s] = s_edge[s][warp + 1];
            if (tid + 1 < T && np == K && q0 + K < N && nxt[s] < r[s][K - 1]) ok = false;
        }
        bool in_order = __syncthreads_and(ok);
        if (C.size > 1) {
            struct Edges {
                R first[2], last[2];
                int flags;
            };
            const Edges* v = C.exchange(Edges{{s_edge[0][0], s_edge[1][0]}, {s_last[0], s_last[1]},
                                              (int)in_order | (stop ? 2 : 0)});
            stop = false;
            Edges before = {};
            for (int i = 0; i < C.size; ++i) {
                const Edges b = C.slot(v, i);
                in_order = in_order && (b.flags & 1) != 0;
                stop = stop || (b.flags & 2) != 0;
                if (i > 0 && i * T * K < N && (b.first[0] < before.last[0] || b.first[1] < before.last[1]))
                    in_order = false;
                before = b;
            }
        }
        if (stop) break;
        stage_radii(W.rho[buf], n, sR);
        if (m <= kRegBeamCap)
            for (int q = tid; q < m; q += T) sB[q] = W.br[b0 + q];
        __syncthreads();
        if (!in_order) {
#pragma unroll 1
            for (int s = 0; s < 2; ++s) {
                RankSort<R> sorter(sR + s * N, N, s_sort);
                sorter.prepare(s_keys);
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < np) {
                        const int p = s * N + sorter.place(q0 + k, s ? r[1][k] : r[0][k]);
                        if (s == 0) store(buf ^ 1, 0, k, p);
                        else store(buf ^ 1, 1, k, p);
                        W.rho_lo[p] = s ? rlo[1][k] : rlo[0][k];
                    }
                __syncthreads();
            }
            buf ^= 1;
            C.sync();
            load();
            stage_radii(W.rho[buf], n, sR);
            __syncthreads();
        }
        const bool staged = m <= kRegBeamCap;
        const R* beamR = staged ? sB : (W.br + b0);
        const bool tables = query || m > 0;

        // ---------------- a3 + a4: beam field at rings; per species own psi, d_rho psi
        R bb[2][K];
        A lnr[2][K];
        Pair<A> loc[2], ex[2], tot[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            loc[s] = zeroP;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                bb[s][k] = 0;
                lnr[s][k] = zeroA;
                if (k < np) {
                    const R x = r[s][k];
                    if (m > 0 && x > (R)0) {
                        const int lb = lower_bound_dev(beamR, m, x);
                        const R Q = lb < m ? W.bE[b0 + lb] : qtot;
                        bb[s][k] = Q * inv_2pi_dxi / x;
                    }
                    lnr[s][k] = ring_log(W.ctab, id[s][k], x, rlo[s][k]);
                    loc[s].x = acc_add_r(loc[s].x, c[s][k]);
                    loc[s].y = acc_add(loc[s].y, acc_mul_r(lnr[s][k], c[s][k]));
                }
            }
        }
        ex[0] = block_excl_scan1<false>(loc[0], OpAddPair(), zeroP, s_ev.w, tot[0]);
        ex[1] = block_excl_scan1<false>(loc[1], OpAddPair(), zeroP, s_w1, tot[1]);
        if (C.size > 1) {
            using Two = TwoVals<Pair<A>, Pair<A>>;
            const Two* v = C.exchange(Two{tot[0], tot[1]});
            if (tid == 0) gm_fold<false>(C, v, zeroP, OpAddPair(), [](Two x) { return x.a; }, s_fold[0], s_fold[1]);
            if (tid == 32 % T)
                gm_fold<false>(C, v, zeroP, OpAddPair(), [](Two x) { return x.b; }, s_fold[2], s_fold[3]);
            __syncthreads();
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                ex[s] = OpAddPair()(s_fold[2 * s], ex[s]);
                tot[s] = s_fold[2 * s + 1];
            }
        }
        A psio[2][K], dpro[2][K];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int rb = s * (N + 1);
            A S = ex[s].x, L = ex[s].y;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    const int p = s * N + q0 + k;
                    const A Lsuf = acc_sub(tot[s].y, L);
                    if (tables) {
                        W.regS[rb + q0 + k] = S;
                        W.regL[rb + q0 + k] = Lsuf;
                    }
                    // own fields kept in the accumulator type: the two species'
                    // values are large and cancel to the small total
                    psio[s][k] = acc_add(Lsuf, acc_mul_a(S, lnr[s][k]));
                    dpro[s][k] = acc_div(acc_add_r(S, ch[s][k]), make_radius(r[s][k], rlo[s][k]));
                    W.psio[p] = psio[s][k];
                    W.dpro[p] = dpro[s][k];
                    W.rho_lo[p] = rlo[s][k];  // (the gathers take radii in the accumulator type)
                    S = acc_add_r(S, c[s][k]);
                    L = acc_add(L, acc_mul_r(lnr[s][k], c[s][k]));
                }
            if (lead && tables) {
                W.regS[rb + N] = tot[s].x;
                W.regL[rb + N] = zeroA;
                W.regT[rb + N] = (R)0;
            }
        }
        C.sync();  // own-species fields, before the other species gathers them

        // ---------------- a5: totals of psi, d_rho psi; psibar, gamma, t
        Locate<A, R> at[2][K];
        R pb[2][K], g[2][K], dpr[2][K], t[2][K], psi[2][K];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int ob = (1 - s) * N;
            const A oS = tot[1 - s].x;
            const A psi_e = acc_mul_a(oS, ln_e), dpr_e = acc_mul_a(oS, inv_e);  // the other species at the edge
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    const R x = r[s][k], v = u[s][k];
                    const A X = make_radius(x, rlo[s][k]);
                    at[s][k] = locate(sR + ob, W.rho_lo + ob, N, edge, Xe, X, x);
                    A psiA, dprA;
                    if (at[s][k].where == 2) {
                        psiA = acc_mul_a(oS, acc_log(X, Xe, ln_e, edge));
                        dprA = acc_div(oS, X);
                    } else {
                        psiA = gather_acc(at[s][k], W.psio + ob, N, tot[1 - s].y, psi_e);
                        dprA = gather_acc(at[s][k], W.dpro + ob, N, zeroA, dpr_e);
                    }
                    psi[s][k] = acc_to_r(acc_add(psio[s][k], psiA));
                    dpr[s][k] = acc_to_r(acc_add(dpro[s][k], dprA));
                    pb[s][k] = (R)1 - qm[s] * psi[s][k];
                    g[s][k] = ((R)1 + v * v + pb[s][k] * pb[s][k]) / ((R)2 * pb[s][k]);
                    t[s][k] = c[s][k] * v / (x * pb[s][k]);
                }
        }

        // ---------------- a6: per species own d_zeta psi, with the electrons' matrices
        A Ttot[2], tl[2], Tex[2];
        R Ac[K], m01[K];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            tl[s] = zeroA;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) tl[s] = acc_add_r(tl[s], t[s][k]);
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) {
                Ac[k] = c[0][k] / r[0][k] / pb[0][k];
                m01[k] = (R)0.5 * Ac[k] / r[0][k];
            }
        const Mat2<R> I2 = {1, 0, 0, 1};
        Mat2<R> Mf, Mb, Yf, Yb, tf, tb;
        ring_products<K>(r[0], Ac, m01, np, Mf, Mb);
        Tex[0] = block_excl_scan_sum_mats1<true>(tl[0], Mf, Mb, zeroA, s_ev.m, Yf, Yb, Ttot[0], tf, tb);
        Tex[1] = block_excl_scan1<false>(tl[1], OpAdd(), zeroA, s_t1, Ttot[1]);
        if (C.size > 1) {
            struct Four {
                A t0, t1;
                Mat2<R> f, r;
            };
            const Four* v = C.exchange(Four{Ttot[0], Ttot[1], tf, tb});
            Mat2<R> all;
            if (tid == 0)
                gm_fold<false>(C, v, I2, OpMatLeft(), [](Four x) { return x.f; }, s_ev.pre_f, all);
            if (tid == 32 % T)
                gm_fold<true>(C, v, I2, OpMatLeft(), [](Four x) { return x.r; }, s_ev.pre_r, all);
            if (tid == 64 % T) {
                gm_fold<false>(C, v, zeroA, OpAdd(), [](Four x) { return x.t0; }, s_tf[0], s_tf[1]);
                gm_fold<false>(C, v, zeroA, OpAdd(), [](Four x) { return x.t1; }, s_tf[2], s_tf[3]);
            }
            __syncthreads();
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                Tex[s] = acc_add(s_tf[2 * s], Tex[s]);
                Ttot[s] = s_tf[2 * s + 1];
            }
            Yf = OpMatLeft()(s_ev.pre_f, Yf);
            Yb = OpMatLeft()(s_ev.pre_r, Yb);
        }
        R dpz[2][K];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int rb = s * (N + 1);
            A Tacc = Tex[s];
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    if (tables) W.regT[rb + q0 + k] = acc_to_r(acc_sub(Ttot[s], Tacc));
                    Tacc = acc_add_r(Tacc, t[s][k]);
                    const R above = acc_to_r(acc_sub(Ttot[s], Tacc));
                    dpz[s][k] = -(above + ((R)1 - ch[s][k] / c[s][k]) * t[s][k]);
                    W.dpzo[s * N + q0 + k] = dpz[s][k];
                }
        }
        C.sync();
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int ob = (1 - s) * N;
            const R oT = acc_to_r(Ttot[1 - s]);
#pragma unroll
            for (int k = 0; k < K; ++k)
                // no ring of the other species above: no d_zeta psi from it
                if (k < np)
                    dpz[s][k] = dpz[s][k] + (at[s][k].where == 2 ? (R)0
                                                                 : gather_r(at[s][k], W.dpzo + ob, N, -oT, (R)0));
        }

        // ---------------- a7 + a8: B_theta^(p) of the electrons (regions 0..N)
        R Bc[K], Cc[K], bp[2][K], bN;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np)
                ring_sources(c[0][k], r[0][k], u[0][k], pb[0][k], g[0][k], dpr[0][k], dpz[0][k], bb[0][k], Bc[k],
                             Cc[k]);
        gm_region_solve<P, K>(W, C, s_ev, N, q0, np, r[0], Ac, m01, Bc, Cc, Yf, Yb, tables, bp[0], bN);
        // B^(p) at the electron rings, then interpolated at the ion rings
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) W.cA[q0 + k] = bp[0][k];
        C.sync();
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np)
                bp[1][k] = at[1][k].where == 2 ? bN / r[1][k] : gather_r(at[1][k], W.cA, N, (R)0, bN / edge);

        // ---------------- guard, dumps
        bool bad = false;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    if (!(pb[s][k] > (R)0) || !real_finite(pb[s][k]) || !real_finite(dpr[s][k]) ||
                        !real_finite(dpz[s][k]) || !real_finite(bp[s][k]) || !real_finite(bb[s][k]) ||
                        !real_finite(g[s][k]))
                        bad = true;
                    if (!query && W.dump_r) {
                        const size_t row = (size_t)slice * n + id[s][k];
                        W.dump_r[row] = r[s][k];
                        if (W.dump_ur) {
                            W.dump_ur[row] = u[s][k];
                            W.dump_psi[row] = psi[s][k];
                            W.dump_dpr[row] = dpr[s][k];
                            W.dump_dpz[row] = dpz[s][k];
                            W.dump_bp[row] = bp[s][k];
                            W.dump_bb[row] = bb[s][k];
                        }
                    }
                }
        bad = wake_vote(C, bad, false);

        // ---------------- a9: fields on beam particles (or query radii)
        if (tables) {
            const int64_t nq = query ? W.nq : (int64_t)m;
            for (int64_t q = gt; q < nq; q += GT) {
                R x;
                if (query) x = (R)W.rq[q];
                else x = staged ? beamR[q] : W.br[b0 + q];
                R psix = 0, dprx = 0, dpzx = 0, bpx = 0, bbx = 0;
                if (x > (R)0) {
                    // the species' enclosed charges and log sums cancel: add
                    // them in the accumulator type before rounding
                    A Ssum = zeroA, Lsum = zeroA;
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const int rb = s * (N + 1);
                        const int k = lower_bound_dev(sR + s * N, N, x);
                        Ssum = acc_add(Ssum, W.regS[rb + k]);
                        Lsum = acc_add(Lsum, W.regL[rb + k]);
                        dpzx -= W.regT[rb + k];
                        if (s == 0) bpx = W.ak[k] * x + W.bk[k] / x;
                    }
                    psix = acc_to_r(acc_add(Lsum, acc_mul_r(Ssum, real_log(x))));
                    dprx = acc_to_r(Ssum) / x;
                    if (!query) {
                        bbx = W.bQs[b0 + q] * inv_2pi_dxi / x;
                    } else if (m > 0) {
                        const int lb = lower_bound_dev(beamR, m, x);
                        const R Q = lb < m ? W.bE[b0 + lb] : qtot;
                        bbx = Q * inv_2pi_dxi / x;
                    }
                } else {
                    psix = acc_to_r(acc_add(W.regL[0], W.regL[N + 1]));
                    dpzx = -(W.regT[0] + W.regT[N + 1]);
                }
                if (!query) {
                    const int64_t o = b0 + q;
                    W.out_ez[o] = -dpzx;
                    W.out_wr[o] = -dprx;
                    W.out_bt[o] = bpx + bbx;
                    W.out_psi[o] = psix;
                } else {
                    if (W.q_ez) W.q_ez[q] = -dpzx;
                    if (W.q_wr) W.q_wr[q] = -dprx;
                    if (W.q_bt) W.q_bt[q] = bpx + bbx;
                    if (W.q_psi) W.q_psi[q] = psix;
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

        // ---------------- a10: AB2 push of both species
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    R gr = u[s][k] / pb[s][k];
                    R gu = -qm[s] * (g[s][k] * dpr[s][k] / pb[s][k] - (bp[s][k] + bb[s][k]));
                    R rn = r[s][k], rl = rlo[s][k], un;
                    if (has_prev) {
                        radius_add(rn, rl, dxi * ((R)1.5 * gr - (R)0.5 * fr[s][k]));
                        un = u[s][k] + dxi * ((R)1.5 * gu - (R)0.5 * fu[s][k]);
                    } else {
                        radius_add(rn, rl, dxi * gr);
                        un = u[s][k] + dxi * gu;
                    }
                    if (rn < (R)0) {  // through the axis: the ring reappears at -rho
                        rn = -rn;
                        rl = -rl;
                        un = -un;
                        gr = -gr;
                        gu = -gu;
                    }
                    r[s][k] = rn;
                    rlo[s][k] = rl;
                    u[s][k] = un;
                    fr[s][k] = gr;
                    fu[s][k] = gu;
                }
        has_prev = 1;
    }
    C.sync();  // (every read of the tables and radii is done)
    if (!query) {
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    store(buf, s, k, s * N + q0 + k);
                    W.rho_lo[s * N + q0 + k] = rlo[s][k];
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

}  // namespace gbwake
