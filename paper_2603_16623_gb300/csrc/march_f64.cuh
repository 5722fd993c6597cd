// march_f64.cuh -- the double-precision march of gridless AB2 wakes: the
// slice chain of march.cuh with the ring state in registers for the whole
// window, one block or a thread-block cluster per wake.
//
// What bounds it: the FP64 pipe.  An FP64 warp instruction holds its
// sub-partition's pipe for 64 cycles, dependent or not (measured: fma, add
// and mul 64, reciprocal 347, the library's log 2054; 1.25 TFLOP/s over 152
// SMs), so what counts is the number of FP64 instructions each of an SM's
// four pipes gets.  The march of march.cuh -- one block per wake, ~590 of
// them per ring and slice, most in divisions and in taking the logarithm
// twice -- took the pipes of one SM: 283 us per slice at 2000 rings.  Here
//   - a wake's rings are split over up to 16 SMs (a cluster), one warp per
//     pipe (f64_shape);
//   - per ring two reciprocals (of rho and psibar) replace the divisions, the
//     logarithm is taken once from a table, the Wronskian of the homogeneous
//     solutions is the constant it is in exact arithmetic (the (0,0) entry of
//     the whole product) instead of a reciprocal per ring, and both solutions
//     are walked as vectors: ~120 FP64 instructions per ring and slice;
//   - order checks, ranks and finiteness tests run on the bit patterns (the
//     integer pipe), and what a scan needs once per block is computed by one
//     warp instead of by every thread.
// Measured on GB300: one wake of 2000 rings 283 -> 26 us per slice; 24 wakes
// of 500-8000 rings in one batch 1013 -> 60 us per slice.  What is left is
// the chain of ~350 FP64 instructions of one warp (a third of them the two
// matrix scans) and five cluster barriers.
// The suffix products of the decaying solution are formed as such (not as
// the total times an inverse prefix, which would cancel), and each thread
// evaluates the region beyond its last ring itself, so B^(p) at the rings
// needs no exchange.  The d_zeta psi sum and the solve's matrices depend on
// psi only and share one exchange: five cluster barriers per slice (the
// order vote, scan 1, scan 2 with the matrices, the Green's sums, the guard).
// State and region tables also go to the wake's global arrays: the radii for
// the ranks and the searches of beam particles, which any thread may serve.
//
// Thread t of the cluster owns the K sorted positions [tK, tK + K); positions
// beyond the last ring hold a ring of zero weight at radius 1, whose sums are
// zero and whose matrix is the identity.
#pragma once

#include "f64_log.cuh"
#include "march.cuh"
#include "rank_sort.cuh"

namespace gbwake {

constexpr int kF64MaxThreads = 256;
constexpr int kF64Warps = kF64MaxThreads / 32;
constexpr int kF64MaxCtas = 16;  // (beyond 8 a non-portable cluster size)
static_assert(kF64MaxCtas <= kMaxPartCtas && kF64MaxCtas <= 16 && kF64Warps <= 16, "one half warp folds them");
constexpr int kF64BeamCap = 1024;  // beam radii of a slice staged in shared memory

// dynamic shared memory for wakes of up to n_max rings
__host__ __device__ inline size_t f64_smem_bytes(int n_max) {
    return (size_t)8 * ((n_max + 1) / 2 * 2 + kF64BeamCap) + RankSort<double>::bytes(n_max);
}

__device__ __forceinline__ bool f64_finite(double x) {
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
// a < b for radii (>= 0) on the integer pipe
__device__ __forceinline__ bool f64_below(double a, double b) { return radius_key(a) < radius_key(b); }

// the logarithm's table, copied to shared memory when a launch starts
static __device__ const F64LogTable kF64LogTable = f64_log_table();

// What the scans leave in shared memory: the warps' and the blocks' totals
// and what one warp makes of them for the others; one per scan of a slice,
// so that none is written again before a later barrier
struct F64Sum2 {
    double warp[2][kF64Warps], blk[2][kF64MaxCtas], pre[2][kF64Warps], tot[2];
};
struct F64Mat {
    double t_warp[kF64Warps], t_blk[kF64MaxCtas], t_pre[kF64Warps], t_tot;
    Mat2<double> warp[kF64Warps], blk[kF64MaxCtas];
    double2 vec[2][kF64Warps];
    double iw;
};

template <class T>
__device__ __forceinline__ T* f64_peer(T* p, int rank) {
    return cooperative_groups::this_cluster().map_shared_rank(p, rank);
}

// Inclusive scans inside each half of a warp (16 lanes, lane order).
__device__ __forceinline__ double f64_half_scan(double v, int at, int steps) {
    for (int o = 1; o < steps; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o, 16);
        if (at >= o) v += u;
    }
    return v;
}
__device__ __forceinline__ Mat2<double> f64_half_scan(Mat2<double> m, int at, int steps) {
    for (int o = 1; o < steps; o <<= 1) {
        const Mat2<double> a = {__shfl_up_sync(0xffffffffu, m.m00, o, 16), __shfl_up_sync(0xffffffffu, m.m01, o, 16),
                                __shfl_up_sync(0xffffffffu, m.m10, o, 16), __shfl_up_sync(0xffffffffu, m.m11, o, 16)};
        if (at >= o) m = OpMatLeft()(a, m);
    }
    return m;
}
__device__ __forceinline__ double f64_half_at(double v, int i) { return __shfl_sync(0xffffffffu, v, i, 16); }

// The exclusive sums over the cluster's threads of x (forward) and of y
// (forward or, REVY, from the last thread); the totals in s.tot.  Two block
// barriers and the cluster's.  Warp 0 folds what the others wait for, its
// lower half x and its upper half y, each lane one warp's or block's total.
template <bool REVY>
__device__ __forceinline__ double2 f64_sum2(const WakeCtas& C, F64Sum2& s, double x, double y) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int half = lane >> 4, at = lane & 15;
    const bool rev = REVY && half;
    const double ix = warp_incl_scan<false>(x, OpAdd()), iy = warp_incl_scan<REVY>(y, OpAdd());
    double ex = shfl_up_t(ix, 1), ey = REVY ? shfl_dn_t(iy, 1) : shfl_up_t(iy, 1);
    if (lane == 0) ex = 0.0;
    if (lane == (REVY ? 31 : 0)) ey = 0.0;
    if (lane == 31) s.warp[0][warp] = ix;
    if (lane == (REVY ? 0 : 31)) s.warp[1][warp] = iy;
    __syncthreads();
    double pre = 0.0;  // warp 0: the sum before warp j (reversed: beyond it)
    const int jw = rev ? nw - 1 - at : at;
    if (warp == 0) {
        const double in = f64_half_scan(at < nw ? s.warp[half][jw] : 0.0, at, nw);
        const double t = f64_half_at(in, nw - 1);
        pre = f64_half_at(in, at > 0 ? at - 1 : 0);
        if (at == 0) pre = 0.0;
        if (C.size == 1) {
            if (at < nw) s.pre[half][jw] = pre;
            if (at == 0) s.tot[half] = t;
        } else if (at < C.size) {
            f64_peer(&s, at)->blk[half][C.rank] = t;
        }
    }
    if (C.size > 1) {
        C.sync();
        if (warp == 0) {
            const int jb = rev ? C.size - 1 - at : at, pos = rev ? C.size - 1 - C.rank : C.rank;
            const double in = f64_half_scan(at < C.size ? s.blk[half][jb] : 0.0, at, C.size);
            const double t = f64_half_at(in, C.size - 1), b = f64_half_at(in, pos > 0 ? pos - 1 : 0);
            if (at < nw) s.pre[half][jw] = pos > 0 ? b + pre : pre;
            if (at == 0) s.tot[half] = t;
        }
    }
    __syncthreads();
    return {s.pre[0][warp] + ex, s.pre[1][warp] + ey};
}

// The exclusive sum of t, and the homogeneous solutions at this thread's
// first and last region from its rings' product M: R (started as (1, 0) on
// the axis) at its first, D (ending as (0, 1) beyond the last ring) at its
// last, both from one exchange.  s.iw: the reciprocal Wronskian.  Warp 0's
// lower half folds forward (columns of the products so far), its upper half
// from the outside in (rows of the products beyond, as the transposed
// matrices' columns in reversed order).
__device__ __forceinline__ double f64_solutions(const WakeCtas& C, F64Mat& s, double t, const Mat2<double>& M,
                                                double2& R, double2& D) {
    const Mat2<double> I2 = {1, 0, 0, 1};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int half = lane >> 4, at = lane & 15;
    // f: products of the lanes up to this one; g: of the lanes from the last
    // down to this one (later rings on the left in both)
    Mat2<double> f = M, g = M;
    double it = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Mat2<double> a = shfl_up_t(f, o), b = shfl_dn_t(g, o);
        const double v = shfl_up_t(it, o);
        if (lane >= o) {
            f = OpMatLeft()(a, f);
            it += v;
        }
        if (lane + o < 32) g = OpMatLeft()(g, b);
    }
    Mat2<double> fe = shfl_up_t(f, 1), ge = shfl_dn_t(g, 1);
    double et = shfl_up_t(it, 1);
    if (lane == 0) {
        fe = I2;
        et = 0.0;
    }
    if (lane == 31) {
        ge = I2;
        s.warp[warp] = f;
        s.t_warp[warp] = it;
    }
    __syncthreads();
    auto half_mat = [&](const Mat2<double>* m, int n) -> Mat2<double> {
        if (at >= n) return I2;
        Mat2<double> v = m[half ? n - 1 - at : at];
        if (half) v = {v.m00, v.m10, v.m01, v.m11};
        return v;
    };
    double pt = 0.0;
    Mat2<double> pw = I2;  // of the warps before (beyond) warp `at` of this half
    if (warp == 0) {
        const Mat2<double> in = f64_half_scan(half_mat(s.warp, nw), at, nw);
        const double ti = f64_half_scan(at < nw ? s.t_warp[at] : 0.0, at, nw);
        const double tt = f64_half_at(ti, nw - 1);
        const int l = nw - 1;
        const Mat2<double> blk = {f64_half_at(in.m00, l), f64_half_at(in.m01, l), f64_half_at(in.m10, l),
                                  f64_half_at(in.m11, l)};
        const int b = at > 0 ? at - 1 : 0;
        const Mat2<double> ex = {f64_half_at(in.m00, b), f64_half_at(in.m01, b), f64_half_at(in.m10, b),
                                 f64_half_at(in.m11, b)};
        const double tb = f64_half_at(ti, b);
        if (at > 0) {
            pw = ex;
            pt = tb;
        }
        if (half == 0 && at < C.size) {
            F64Mat* to = C.size > 1 ? f64_peer(&s, at) : &s;
            to->blk[C.rank] = blk;
            to->t_blk[C.rank] = tt;
        }
        __syncwarp();
    }
    if (C.size > 1) C.sync();
    if (warp == 0) {
        const Mat2<double> in = f64_half_scan(half_mat(s.blk, C.size), at, C.size);
        const double ti = f64_half_scan(at < C.size ? s.t_blk[at] : 0.0, at, C.size);
        const int l = C.size - 1, pos = half ? l - C.rank : C.rank, b = pos > 0 ? pos - 1 : 0;
        double2 v = {f64_half_at(in.m00, b), f64_half_at(in.m10, b)};
        double bt = f64_half_at(ti, C.rank > 0 ? C.rank - 1 : 0);
        const double tt = f64_half_at(ti, l), w = f64_half_at(in.m00, l);
        if (pos == 0) v = {1.0, 0.0};
        if (C.rank == 0) bt = 0.0;
        if (at < nw)
            s.vec[half][half ? nw - 1 - at : at] = {fma(pw.m00, v.x, pw.m01 * v.y), fma(pw.m10, v.x, pw.m11 * v.y)};
        if (lane < nw) s.t_pre[lane] = bt + pt;
        if (lane == 0) {
            s.t_tot = tt;
            s.iw = __drcp_rn(w);
        }
    }
    __syncthreads();
    const double2 v = s.vec[0][warp], w = s.vec[1][warp];
    R = {fma(fe.m00, v.x, fe.m01 * v.y), fma(fe.m10, v.x, fe.m11 * v.y)};
    // D = (product beyond)^-1 (0, 1) = (-m01, m00), det = 1
    D = {-fma(w.x, ge.m01, w.y * ge.m11), fma(w.x, ge.m00, w.y * ge.m10)};
    return s.t_pre[warp] + et;
}

template <int K>
__global__ void __launch_bounds__(kF64MaxThreads)
march_f64_kernel(const WakeDev<PrecF64>* __restrict__ wakes, const int32_t* __restrict__ order, int32_t max_slices,
                 int32_t mode) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ctl[CTL_N];
    __shared__ int s_stop;
    __shared__ __align__(16) unsigned char s_part[2 * kPartBuf];
    __shared__ double s_edge[kF64Warps];
    __shared__ int64_t s_keys[64];
    __shared__ F64Sum2 s_w, s_g;
    __shared__ F64Mat s_m;
    __shared__ F64LogTable s_log;

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
    const WakeDev<PrecF64>& W = wakes[order ? order[wi] : wi];
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = W.n, n_steps = W.n_steps;
    const int p0 = min(n, (C.rank * T + tid) * K);
    const int np = min(K, n - p0);  // rings this thread holds
    const bool lead = C.rank == 0 && tid == 0;

    double* sR = reinterpret_cast<double*>(smem);  // all radii (staged when searched)
    double* sB = sR + (n + 1) / 2 * 2;             // the slice's beam radii
    RankSort<double> sorter(sR, n, sB + kF64BeamCap);

    if (tid < CTL_N) s_ctl[tid] = W.ctl[tid];
    __syncthreads();
    if (s_ctl[CTL_STATUS] != 0) return;
    int slice = s_ctl[CTL_NEXT];
    int buf = s_ctl[CTL_BUF];
    int has_prev = s_ctl[CTL_PREV];
    int status = 0, fail = -1;
    const int s_end = mode == MODE_MARCH ? min(n_steps, slice + max_slices) : slice + 1;

    const double rmax = W.rho_max, half_n = 0.5 * W.density, quarter_n = 0.25 * W.density;
    const double Imax = half_n * rmax * rmax;
    const double c0 = 0.25 * W.density * rmax * rmax - 0.5 * W.density * rmax * rmax * log(rmax);
    const double dxi = W.dxi;
    const double inv_2pi_dxi = 1.0 / (6.283185307179586476925286766559 * W.dxi);

    double r[K], u[K], fr[K], fu[K], w[K], wh[K];
    int id[K];
    auto load = [&]() {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int p = p0 + k;
            const bool on = k < np;
            r[k] = on ? W.rho[buf][p] : 1.0;
            u[k] = on ? W.ur[buf][p] : 0.0;
            fr[k] = on ? W.frho[buf][p] : 0.0;
            fu[k] = on ? W.fur[buf][p] : 0.0;
            id[k] = on ? W.rid[buf][p] : 0;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            w[k] = k < np ? W.w[id[k]] : 0.0;
            wh[k] = k < np ? W.wh[id[k]] : 0.0;
        }
    };
    auto store = [&](int b, int k, int p) {
        W.rho[b][p] = r[k];
        W.ur[b][p] = u[k];
        W.frho[b][p] = fr[k];
        W.fur[b][p] = fu[k];
        W.rid[b][p] = id[k];
    };
    load();
    for (int i = tid; i < 3 * kLogCells; i += T)
        reinterpret_cast<double*>(&s_log)[i] = reinterpret_cast<const double*>(&kF64LogTable)[i];
    __syncthreads();

    // the beam offsets of this slice and the next, loaded one slice ahead
    const bool beam = W.nb > 0;
    int o0 = 0, o1 = 0;
    double qtot = 0.0;
    if (beam && slice < n_steps) {
        o0 = W.boff[slice];
        o1 = W.boff[slice + 1];
        qtot = W.bTot[slice];
    }

    const int slice0 = slice;
    uint64_t t_start = 0;
    for (; slice < s_end; ++slice) {
        if (W.budget_ns > 0 && tid == 0) {  // (read after the order check's barriers)
            const uint64_t now = global_ns();
            if (slice == slice0) t_start = now;
            s_stop = slice > slice0 && now - t_start >= (uint64_t)W.budget_ns;
        }
        // ---------------- a2: order check; the ranks and the move of rings that crossed
        bool ok = true;
#pragma unroll
        for (int k = 1; k < K; ++k)
            if (k < np && f64_below(r[k], r[k - 1])) ok = false;
        double nxt = shfl_dn_t(r[0], 1);
        if (lane == 0) s_edge[warp] = r[0];
        __syncthreads();
        if (lane == 31 && tid + 1 < T) nxt = s_edge[warp + 1];
        if (tid + 1 < T && np == K && p0 + K < n && f64_below(nxt, r[K - 1])) ok = false;
        bool in_order = __syncthreads_and(ok);
        bool stop = W.budget_ns > 0 && s_stop;
        if (C.size > 1) {  // the blocks agree on both, and on the order across their edges
            struct Edge {
                double first, last;
                int flags;
            };
            Edge e = {r[0], 0.0, (int)in_order | (stop ? 2 : 0)};
            // (the block's last radius: its last ring's owner's)
            __shared__ double s_last;
            if (np > 0 && (tid == T - 1 || p0 + np == n)) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k == np - 1) s_last = r[k];
            }
            __syncthreads();
            e.first = s_edge[0];
            e.last = s_last;
            const Edge* v = C.exchange(e);
            in_order = true;
            stop = false;
            for (int i = 0; i < C.size; ++i) {
                const Edge b = C.slot(v, i);
                in_order = in_order && (b.flags & 1) != 0;
                stop = stop || (b.flags & 2) != 0;
                if (i > 0 && i * T * K < n && f64_below(b.first, C.slot(v, i - 1).last)) in_order = false;
            }
        }
        if (stop) break;
        const int b0 = o0, m = o1 - o0;
        const double qt = qtot;
        if (beam) {
            o0 = o1;
            if (slice + 1 < n_steps) {
                o1 = W.boff[slice + 2];
                qtot = W.bTot[slice + 1];
            }
        }
        const bool query = mode != MODE_MARCH;
        if (!in_order) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];
            C.sync();
            for (int p = tid; p < n; p += T) sR[p] = W.rho[buf][p];
            __syncthreads();
            sorter.prepare(s_keys);
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) store(buf ^ 1, k, sorter.place(p0 + k, r[k]));
            buf ^= 1;
            C.sync();
            load();
        } else if (m > 0 || query) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) W.rho[buf][p0 + k] = r[k];
            // (read after the barriers of the scans)
        }

        // ---------------- a3: the beam's charge inside each ring
        double bb[K], ir[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            ir[k] = __drcp_rn(r[k]);
            bb[k] = 0.0;
        }
        if (m > 0) {
            const double* br = W.br + b0;
            if (m <= kF64BeamCap) {
                for (int q = tid; q < m; q += T) sB[q] = br[q];
                __syncthreads();
                br = sB;
            }
            int lb = 0;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np) {
                    // (radii only grow along the thread's rings)
                    int lo = lb, hi = m;
                    if (k > 0 && (lo >= m || !f64_below(br[lo], r[k]))) hi = lo;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (f64_below(br[mid], r[k])) lo = mid + 1;
                        else hi = mid;
                    }
                    lb = lo;
                    const double Q = lb < m ? W.bE[b0 + lb] : qt;
                    bb[k] = r[k] > 0.0 ? Q * inv_2pi_dxi * ir[k] : 0.0;
                }
        }

        // ---------------- a4: sums of (w, w ln rho)
        double lnr[K], sw = 0.0, sl = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            lnr[k] = k < np ? f64_log(s_log, r[k]) : 0.0;
            sw += w[k];
            sl = fma(w[k], lnr[k], sl);
        }
        const double2 ex = f64_sum2<false>(C, s_w, sw, sl);
        const double Wtot = s_w.tot[0], Ltot = s_w.tot[1];

        // ---------------- a5: psi, d_rho psi, psibar, gamma, t; the solve's matrices
        // (the jump matrix of a ring is I + h (1, -r^2)^T (r, 1/r), its inverse
        // the same with -h: a vector is taken across it in four operations)
        double pb[K], ipb[K], dpr[K], gi[K], t[K], uir[K], hA[K], hr[K], hi[K], psi[K];
        Mat2<double> M = {1, 0, 0, 1};
        double S = ex.x, L = ex.y, tl = 0.0;
        const bool tables = m > 0 || query;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double Ls = Ltot - L, r2 = r[k] * r[k];
            const bool inside = f64_below(r[k], rmax);
            const double Ir = inside ? half_n * r2 : Imax;
            // (at rho = rho_max both forms of the ion potential are equal)
            const double pion = inside ? fma(-quarter_n, r2, c0) : -Imax * lnr[k];
            psi[k] = fma(S, lnr[k], Ls) + pion;
            dpr[k] = (S + wh[k] - Ir) * ir[k];
            pb[k] = k < np ? 1.0 + psi[k] : 1.0;
            ipb[k] = __drcp_rn(pb[k]);
            const double up = u[k] * ipb[k];
            // gamma / psibar
            gi[k] = 0.5 * fma(up, up, fma(ipb[k], ipb[k], 1.0));
            uir[k] = up * ir[k];
            t[k] = w[k] * uir[k];
            tl += t[k];
            hA[k] = 0.5 * (w[k] * ir[k]) * ipb[k];
            hr[k] = hA[k] * r[k];
            hi[k] = hA[k] * ir[k];
            if (k == 0) {
                M = {1.0 + hr[k], hi[k], -hr[k] * r2, 1.0 - hr[k]};
            } else {
                const double q0 = fma(hr[k], M.m00, hi[k] * M.m10), q1 = fma(hr[k], M.m01, hi[k] * M.m11);
                M = {M.m00 + q0, M.m01 + q1, fma(-r2, q0, M.m10), fma(-r2, q1, M.m11)};
            }
            if (tables && k < np) {
                W.regS[p0 + k] = S;
                W.regL[p0 + k] = Ls;
            }
            S += w[k];
            L = fma(w[k], lnr[k], L);
        }
        double2 Rv, Dv;
        const double Tex = f64_solutions(C, s_m, tl, M, Rv, Dv);
        const double Ttot = s_m.t_tot, iw = s_m.iw;

        // ---------------- a6 + a7: d_zeta psi, ring sources; the walks of R and D
        double dpz[K], s0[K], s1[K], R0[K + 1], R1[K + 1], D0[K + 1], D1[K + 1];
        R0[0] = Rv.x;
        R1[0] = Rv.y;
        {
            double Ta = Tex;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (tables && k < np) W.regT[p0 + k] = Ttot - Ta;
                Ta += t[k];
                dpz[k] = -fma(w[k] - wh[k], uir[k], Ttot - Ta);
                const double up = u[k] * ipb[k], c = fma(up, up, -gi[k]);
                const double A = 2.0 * hA[k];
                const double B = A * fma(-up, dpz[k], fma(dpr[k], c, fma(ir[k] * u[k], up, bb[k])));
                const double Cc = w[k] * ir[k] * (1.0 + c);
                s0[k] = 0.5 * fma(hA[k], Cc, B);
                s1[k] = r[k] * fma(-r[k], s0[k], Cc);
                const double q = fma(hr[k], R0[k], hi[k] * R1[k]);
                R0[k + 1] = R0[k] + q;
                R1[k + 1] = fma(-(r[k] * r[k]), q, R1[k]);
            }
        }
        D0[K] = Dv.x * iw;
        D1[K] = Dv.y * iw;
        double gp[K], dp[K], gl = 0.0, dl = 0.0;
#pragma unroll
        for (int k = K - 1; k >= 0; --k) {
            gp[k] = fma(s0[k], D1[k + 1], -s1[k] * D0[k + 1]);  // (D carries 1 / Wronskian)
            dp[k] = fma(R0[k + 1], s1[k], -R1[k + 1] * s0[k]);
            gl += gp[k];
            dl += dp[k];
            const double q = fma(hr[k], D0[k + 1], hi[k] * D1[k + 1]);
            D0[k] = D0[k + 1] - q;
            D1[k] = fma(r[k] * r[k], q, D1[k + 1]);
        }
        const double2 gd = f64_sum2<true>(C, s_g, dl, gl);

        // ---------------- a8: the regions' a, b; B^(p) at the rings, guard, dumps
        double a[K + 1], b[K + 1], bp[K];
        {
            double G = gd.y, H = gd.x;
            a[K] = -G * R0[K];
            b[K] = -G * R1[K];
#pragma unroll
            for (int k = K - 1; k >= 0; --k) {
                G += gp[k];
                a[k] = -G * R0[k];
                b[k] = -G * R1[k];
            }
#pragma unroll
            for (int k = 0; k <= K; ++k) {
                a[k] = fma(H, D0[k], a[k]);
                b[k] = fma(H, D1[k], b[k]);
                if (k < K) H += dp[k];
            }
        }
        bool bad = false;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            bp[k] = 0.5 * fma(a[k] + a[k + 1], r[k], (b[k] + b[k + 1]) * ir[k]);
            if (k < np) {
                const int p = p0 + k;
                if (!(pb[k] > 0.0) || !f64_finite(pb[k]) || !f64_finite(dpr[k]) || !f64_finite(dpz[k]) ||
                    !f64_finite(bp[k]) || !f64_finite(bb[k]) || !f64_finite(gi[k]))
                    bad = true;
                if (tables) {
                    W.ak[p] = a[k];
                    W.bk[p] = b[k];
                    if (p == n - 1) {  // beyond the last ring
                        W.ak[n] = a[k + 1];
                        W.bk[n] = b[k + 1];
                    }
                }
                if (!query && W.dump_r) {
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
        }
        if (tables && lead) {
            W.regS[n] = Wtot;
            W.regL[n] = 0.0;
            W.regT[n] = 0.0;
        }
        if (tables)  // the radii, stored before the scans' barriers
            for (int p = tid; p < n; p += T) sR[p] = W.rho[buf][p];
        bad = wake_vote(C, bad, false);

        // ---------------- a9: fields on beam particles (or query radii)
        if (tables) {
            const int64_t nq = query ? W.nq : (int64_t)m;
            // warps of 32 particles go round the blocks, so that a short
            // slice's work spreads over their FP64 pipes
            const int64_t GT = (int64_t)C.size * T;
            for (int64_t q = ((int64_t)warp * C.size + C.rank) * 32 + lane; q < nq; q += GT) {
                const double x = query ? W.rq[q] : m <= kF64BeamCap ? sB[q] : W.br[b0 + q];
                double psi_x, dprx, dpzx, bpx, bbx;
                if (x > 0.0) {
                    const int k = lower_bound_dev(reinterpret_cast<const int64_t*>(sR), n, radius_key(x));
                    const double ix = __drcp_rn(x), lnx = f64_log(s_log, x), x2 = x * x;
                    const double Sk = W.regS[k];
                    const bool inside = x < rmax;
                    const double pion = x <= rmax ? c0 - x2 * quarter_n : Imax * -lnx;
                    psi_x = fma(Sk, lnx, W.regL[k]) + pion;
                    dprx = (Sk - (inside ? half_n * x2 : Imax)) * ix;
                    dpzx = -W.regT[k];
                    bpx = W.ak[k] * x + W.bk[k] * ix;
                    if (!query) {
                        bbx = W.bQs[b0 + q] * inv_2pi_dxi * ix;
                    } else {
                        bbx = 0.0;
                        if (m > 0) {
                            const int l2 = lower_bound_dev(W.br + b0, m, x);
                            bbx = (l2 < m ? W.bE[b0 + l2] : qt) * inv_2pi_dxi * ix;
                        }
                    }
                } else {
                    psi_x = W.regL[0] + c0;
                    dprx = 0.0;
                    dpzx = -W.regT[0];
                    bpx = 0.0;
                    bbx = 0.0;
                }
                if (!query) {
                    const int64_t o = b0 + q;
                    W.out_ez[o] = -dpzx;
                    W.out_wr[o] = -dprx;
                    W.out_bt[o] = bpx + bbx;
                    W.out_psi[o] = psi_x;
                } else {
                    if (W.q_ez) W.q_ez[q] = -dpzx;
                    if (W.q_wr) W.q_wr[q] = -dprx;
                    if (W.q_bt) W.q_bt[q] = bpx + bbx;
                    if (W.q_psi) W.q_psi[q] = psi_x;
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

        // ---------------- a10: AB2 push
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double gr = u[k] * ipb[k], gu = fma(gi[k], dpr[k], -(bp[k] + bb[k]));
            const double dr = has_prev ? fma(1.5, gr, -0.5 * fr[k]) : gr;
            const double du = has_prev ? fma(1.5, gu, -0.5 * fu[k]) : gu;
            double rn = k < np ? fma(dxi, dr, r[k]) : 1.0, un = k < np ? fma(dxi, du, u[k]) : 0.0;
            if (__double2hiint(rn) < 0) {  // through the axis: the ring reappears at -rho
                rn = -rn;
                un = -un;
                gr = -gr;
                gu = -gu;
            }
            r[k] = rn;
            u[k] = un;
            fr[k] = gr;
            fu[k] = gu;
        }
        has_prev = 1;
    }
    C.sync();  // (every read of the tables and radii is done)
    if (mode == MODE_MARCH) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < np) store(buf, k, p0 + k);
    }
    if (lead) {
        if (mode == MODE_MARCH) put_march_times(W.ctl, t_launch);
        W.ctl[CTL_NEXT] = mode == MODE_MARCH ? slice : s_ctl[CTL_NEXT];
        W.ctl[CTL_BUF] = buf;
        W.ctl[CTL_PREV] = has_prev;
        if (status) {
            W.ctl[CTL_STATUS] = status;
            W.ctl[CTL_FAIL] = fail;
        }
    }
}

}  // namespace gbwake
