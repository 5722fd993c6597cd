// march_cluster.cuh -- the on-chip march of one wake by a thread-block
// cluster: CTA c of the cluster holds the sorted ring positions
// [c*T*K, (c+1)*T*K) in its shared memory (same layout as march_fast.cuh).
// The per-slice chain is that of march_fast.cuh; what crosses CTAs goes
// through distributed shared memory, pushed by remote stores into each
// peer's receive slots and read locally after one cluster barrier:
//   - the sortedness vote, every CTA's first and last radius and the guard
//     of the previous slice (one exchange at the top of each slice; the AB2
//     push of a slice waits in the dead region-table arrays and becomes the
//     state only if no CTA failed the guard);
//   - the block-scan totals (each CTA folds the totals of its predecessors,
//     or successors for the reverse scans, in rank order: deterministic): the
//     sums of w and w ln rho, the sum of t with the two matrix products, and
//     the two Green's-function sums, one exchange each;
//   - the region table entry just past each CTA's last ring.
// Every ring finds its place among the slice's beam radii, and the fields on
// beam particles stay inside each CTA: each takes the particles (or query
// radii) between the previous CTA's last radius and its own, whose rings and
// regions it holds.  When rings crossed, every CTA sorts its own range and
// the rings that belong to another CTA are counted and moved there.
// Every cluster barrier is reached in cluster-uniform control flow.
#pragma once

#include <cooperative_groups.h>

#include "march_fast.cuh"

namespace gbwake {

namespace cg = cooperative_groups;

template <class T>
__device__ __forceinline__ T* rmt(cg::cluster_group& cl, T* p, int rank) {
#ifdef WAKE_BOUNDS_CHECK
    rank = bounds_checked(rank, (int)cl.num_blocks());
#endif
    return cl.map_shared_rank(p, rank);
}

__device__ __forceinline__ FastSmem rmt_sm(cg::cluster_group& cl, const FastSmem& s, int r) {
    FastSmem o;
    o.rh = rmt(cl, s.rh, r);
    o.rl = rmt(cl, s.rl, r);
    o.u = rmt(cl, s.u, r);
    o.fr = rmt(cl, s.fr, r);
    o.fu = rmt(cl, s.fu, r);
    o.id = rmt(cl, s.id, r);
    o.a = rmt(cl, s.a, r);
    o.b = rmt(cl, s.b, r);
    o.T = rmt(cl, s.T, r);
    o.D = rmt(cl, s.D, r);
    o.S = rmt(cl, s.S, r);
    o.psi = rmt(cl, s.psi, r);
    return o;
}

// Push of one value per CTA: every CTA stores v into slot [its rank] of
// each peer's recv array (threads 0..size-1, one peer each).  The values are
// read after the next cluster barrier.
template <class T>
__device__ __forceinline__ void cluster_push(cg::cluster_group& cl, T* recv, const T& v) {
    const int rank = cl.block_rank(), size = cl.num_blocks();
    if ((int)threadIdx.x < size) *rmt(cl, &recv[rank], threadIdx.x) = v;
}

// Folds of the received totals in rank order: over ranks < mine (pre) and
// over all ranks (all).  Every thread computes them from shared memory.
template <class T, class Op>
__device__ __forceinline__ void fold_fwd(const T* recv, int rank, int size, T ident, Op op, T& pre, T& all) {
    pre = ident;
    all = ident;
    for (int r = 0; r < size; ++r) {
        if (r == rank) pre = all;
        all = op(all, recv[r]);
    }
}

// the same for a reverse scan: over ranks > mine, from the last rank down
template <class T, class Op>
__device__ __forceinline__ void fold_rev(const T* recv, int rank, int size, T ident, Op op, T& pre, T& all) {
    pre = ident;
    all = ident;
    for (int r = size - 1; r >= 0; --r) {
        if (r == rank) pre = all;
        all = op(all, recv[r]);
    }
}

// The forward fold by thread 0 into shared memory, read by every thread after
// a block barrier (keeps the fold's registers out of the callers' peak).
template <class T, class Op>
__device__ __forceinline__ void fold_fwd_shared(const T* recv, int rank, int size, T ident, Op op, T* s_pre,
                                                T* s_all) {
    if (threadIdx.x == 0) {
        T pre, all;
        fold_fwd(recv, rank, size, ident, op, pre, all);
        *s_pre = pre;
        *s_all = all;
    }
    __syncthreads();
}

// shared memory of the cluster march: the fast march's arrays plus one for
// cluster_move's copies of other CTAs' radii
__host__ __device__ inline size_t cluster_smem_bytes(int T, int K) {
    return fast_smem_bytes(T, K) + 4 * ((size_t)T * K + 8);
}

// block-uniform: are the radii rh (this CTA's rings) in order?
template <int K>
__device__ __forceinline__ bool block_sorted(const float* rh, int nl, int p0) {
    using SW = Swz<K>;
    bool ok = true;
    float prev = -INFINITY;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int p = p0 + k;
        if (p < nl) {
            float v = rh[SW::at(p)];
            if (v < prev) ok = false;
            prev = v;
        }
    }
    if (p0 + K < nl && rh[SW::at(p0 + K)] < prev) ok = false;
    return __syncthreads_and(ok);
}

// Moves every ring to its place in the cluster's order, each CTA's own range
// being sorted already (and without NaN: the places are then a permutation).
// A ring's place is its position, less the rings of the CTAs before that lie
// above it, plus the rings of the CTAs after that lie below it (equal radii
// keep their order, which keeps the sort stable).  Those rings are the last
// of an earlier CTA's range, the first of a later one's: a warp per CTA finds
// how many concern this CTA (32 probes at a time, at most 3 too many), their
// radii are copied to `scratch` (TK words, as many CTAs at a time as fit) and
// searched there.  The rings are then written to their place in the owner's
// dead region tables, read back after the one cluster barrier.  Bound by
// latency (remote loads, barriers): odd-even merge rounds between neighbours,
// each moving every ring through two cluster barriers, took 24.8k cycles of a
// 74k-cycle slice with the blocks' own sorts (6000 warm rings on 6 blocks),
// this 17.2k: the warm restart 5.62 -> 5.21 ms, 65,536 rings 17.7 -> 17.3 ms.
// s_edges: every CTA's first and last radius; s_last: receives the last
// radius every CTA then holds.
template <int K>
__device__ void cluster_move(cg::cluster_group& cl, const FastSmem& sm, int n, int TK, int nl, float* scratch,
                             const float2* s_edges, int* s_cnt, float* s_last) {
    using SW = Swz<K>;
    const int rank = cl.block_rank(), size = cl.num_blocks();
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, nw = T >> 5;
    for (int r = tid >> 5; r < size; r += nw) {
        const bool before = r < rank;
        const float x = before ? s_edges[rank].x : s_edges[rank].y;
        int c = 0;
        if (r != rank && (before ? s_edges[r].y > x : s_edges[r].x < x)) {
            const int nr = min(TK, n - r * TK);
            const float* rh = rmt(cl, sm.rh, r);
            int len = nr - 1;
            c = 1;  // the count lies in [c, c + len]
#pragma unroll
            for (int round = 0; round < 2; ++round) {
                const int step = max(1, (len + 31) / 32), i = c + (lane + 1) * step - 1;
                bool out = false;  // does ring i, counted from the near end, lie beyond x?
                if (i < c + len) {
                    const float v = rh[SW::at(before ? nr - 1 - i : i)];
                    out = before ? v > x : v < x;
                }
                const int some = __popc(__ballot_sync(0xffffffffu, out)) * step;
                c += some;
                len = min(step - 1, len - some);
            }
            c += len;
        }
        if (lane == 0) s_cnt[r] = c;
    }
    __syncthreads();
    const int p0 = tid * K, np = max(0, min(K, nl - p0));
    float x[K];
    int place[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        x[k] = k < np ? sm.rh[SW::at(p0 + k)] : INFINITY;
        place[k] = rank * TK + p0 + k;
    }
    for (int r0 = 0; r0 < size;) {
        int r1 = r0, total = 0;
        while (r1 < size && total + s_cnt[r1] <= TK) total += s_cnt[r1++];  // (a count is at most TK)
        for (int i = tid; i < total; i += T) {
            int r = r0, o = i;
            while (o >= s_cnt[r]) o -= s_cnt[r++];
            const int at = r < rank ? min(TK, n - r * TK) - s_cnt[r] + o : o;
            scratch[i] = rmt(cl, sm.rh, r)[SW::at(at)];
        }
        __syncthreads();
        const float* seg = scratch;
        for (int r = r0; r < r1; ++r) {
            const int c = s_cnt[r];
            const bool before = r < rank;
            bool any = false;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < np && (before ? x[k] < s_edges[r].y : x[k] > s_edges[r].x)) any = true;
            if (c > 0 && any) {
                int lo[K];  // how many of the segment lie below x (or at x, before)
#pragma unroll
                for (int k = 0; k < K; ++k) lo[k] = 0;
                for (int len = c; len > 0;) {
                    const int h = (len + 1) >> 1;
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        const float v = seg[lo[k] + h - 1];
                        if (before ? v <= x[k] : v < x[k]) lo[k] += h;
                    }
                    len -= h;
                }
#pragma unroll
                for (int k = 0; k < K; ++k) place[k] += before ? lo[k] - c : lo[k];
            }
            seg += c;
        }
        r0 = r1;
        if (r0 < size) __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (k < np) {
            const int a = SW::at(p0 + k), r = place[k] / TK, l = place[k] - r * TK, to = SW::at(l);
            *rmt(cl, &sm.a[to], r) = x[k];
            *rmt(cl, &sm.b[to], r) = sm.rl[a];
            *rmt(cl, &sm.T[to], r) = sm.u[a];
            *rmt(cl, &sm.D[to], r) = sm.fr[a];
            *rmt(cl, &sm.S[to], r) = sm.fu[a];
            *rmt(cl, &sm.psi[to], r) = __int_as_float(sm.id[a]);
            if (l == min(TK, n - r * TK) - 1)
                for (int q = 0; q < size; ++q) *rmt(cl, &s_last[r], q) = x[k];
        }
    }
    cl.sync();  // every ring has arrived, every read of the old ranges is done
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (k < np) {
            const int a = SW::at(p0 + k);
            sm.rh[a] = sm.a[a];
            sm.rl[a] = sm.b[a];
            sm.u[a] = sm.T[a];
            sm.fr[a] = sm.D[a];
            sm.fu[a] = sm.S[a];
            sm.id[a] = __float_as_int(sm.psi[a]);
        }
    }
}

template <int K>
__global__ void __launch_bounds__(512)
march_cluster_kernel(const WakeDev<PrecMixed>* __restrict__ wakes, const int32_t* __restrict__ order,
                     int32_t max_slices, int32_t mode, int32_t stage_particles) {
    using R = float;
    using A = ff;
    using SW = Swz<K>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ctl[CTL_N];
    __shared__ float4 s_xch[16];   // per rank: (in order?, first radius, last radius, failed the guard?)
    __shared__ float s_last[16];   // last radius held by every CTA, this slice
    __shared__ float2 s_edges[16];  // every CTA's first and last radius after its own sort
    __shared__ int s_cnt[16];       // rings of every CTA that cross this CTA's edges
    __shared__ int s_stop;
    __shared__ float2 s_nab;       // (a, b) of the next CTA's first region
    __shared__ Pair<ff> x1[16], f1[2];
    __shared__ ff x2[16], f2[2];
    __shared__ Mat2<float> x3f[16], x3r[16], f3[4];
    __shared__ ff x4f[16], x4r[16], f4[4];
    __shared__ __align__(8) uint64_t s_bar[2];

    cg::cluster_group cl = cg::this_cluster();
    const int crank = cl.block_rank();
    const int csize = cl.num_blocks();
    const int widx = blockIdx.x / csize;
    const uint64_t t_launch = global_ns();
    // a query (one wake): every cluster solves the slice and takes its share of the radii
    const WakeDev<PrecMixed>& W = wakes[mode == MODE_QUERY ? 0 : order ? order[widx] : widx];
    const int T = blockDim.x;
    const int tid = threadIdx.x;
    const int n = W.n;
    const int TK = T * K;
    const int base = crank * TK;               // global position of local slot 0
    const int nl = max(0, min(TK, n - base));  // rings held by this CTA (>= 1)
    const int p0 = tid * K;                    // local positions [p0, p0 + K)
    const int nv = nl - p0;                    // of them the first nv hold rings
    const int cap = TK + 8;
    const bool last_cta = crank == csize - 1;  // holds the last ring and region n
    const RingTab ctab = W.ctab;

    unsigned char* sscan = smem;
    FastSmem sm;
    sm.rh = reinterpret_cast<float*>(smem + kScanBytes);
    sm.rl = sm.rh + cap;
    sm.u = sm.rl + cap;
    sm.fr = sm.u + cap;
    sm.fu = sm.fr + cap;
    sm.id = reinterpret_cast<int32_t*>(sm.fu + cap);
    sm.a = reinterpret_cast<float*>(sm.id + cap);
    sm.b = sm.a + cap;
    sm.T = sm.b + cap;
    sm.D = sm.T + cap;
    sm.S = sm.D + cap;
    sm.psi = sm.S + cap;
    float* scratch = sm.psi + cap;  // cluster_move's copies of other CTAs' radii

    if (tid < CTL_N) s_ctl[tid] = W.ctl[tid];
    cl.sync();  // every CTA has started before any stores into another's shared memory
    // (status and slice are the same for every CTA of the cluster)
    if (s_ctl[CTL_STATUS] != 0) return;
    int slice = s_ctl[CTL_NEXT];
    const int buf = s_ctl[CTL_BUF];
    int has_prev = s_ctl[CTL_PREV];
    int status = 0, fail = -1;
    const int n_steps = W.n_steps;
    const int s_end = mode == MODE_MARCH ? min(n_steps, slice + max_slices) : slice + 1;

    for (int p = tid; p < nl; p += T) {
        int a = SW::at(p), g = base + p;
        sm.rh[a] = W.rho[buf][g];
        sm.rl[a] = W.rho_lo[g];
        sm.u[a] = W.ur[buf][g];
        sm.fr[a] = W.frho[buf][g];
        sm.fu[a] = W.fur[buf][g];
        sm.id[a] = W.rid[buf][g];
    }
    __syncthreads();

    const double dens_d = W.density, rmax_d = W.rho_max;
    const R rmax = (R)rmax_d;
    const R half_n = (R)(0.5 * dens_d), quarter_n = (R)(0.25 * dens_d);
    const A Imax = ff_from_d(0.5 * dens_d * rmax_d * rmax_d);
    const A c0 = ff_from_d(0.25 * dens_d * rmax_d * rmax_d - 0.5 * dens_d * rmax_d * rmax_d * log(rmax_d));
    const R dxi = (R)W.dxi;
    const R inv_2pi_dxi = (R)(1.0 / (6.283185307179586476925286766559 * W.dxi));
    const A zeroA = {0.f, 0.f};
    const Mat2<R> I2 = {1, 0, 0, 1};

    // beam stage (march only): every CTA stages the whole slice after its
    // ring arrays and its count array
    BeamStage stg;
    stg.base = reinterpret_cast<float*>(smem + cluster_smem_bytes(T, K));
    stg.bar = s_bar;
    stg.cap = (mode == MODE_MARCH && W.nb > 0 && (W.stage & STAGE_OK)) ? stage_cap_floats(stage_particles) : 0;
    // test only: the first slice staged during the march is never copied
    bool stall_armed = (W.stage & STAGE_TEST_STALL) != 0;
    if (stg.cap > 0 && tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        mbar_fence_init();
    }
    uint32_t parity = 0;  // per buffer: the phase its next wait completes
    int pending = 0;      // per buffer: a staged copy not yet waited for
    __syncthreads();
    if (stg.cap > 0 && slice < n_steps &&
        stage_slice(stg, W, slice, W.boff[slice], W.boff[slice + 1] - W.boff[slice], false))
        pending |= 1 << (slice & 1);

    R rh[K], ur[K];
    int idv[K];
    R ir[K], ipb[K];
    R pbv[K], dprv[K], bbv[K];
    R s0v[K], s1v[K], hav[K];
    R tv[K];
    // at 8 rings per thread recomputed where used (the same rounding: the
    // same reciprocal of the same value), which keeps 16 registers free
    auto IR = [&](int k) -> R {
        if constexpr (K >= 8) return __frcp_rn(rh[k]);
        else return ir[k];
    };
    auto IPB = [&](int k) -> R {
        if constexpr (K >= 8) return __frcp_rn(pbv[k]);
        else return ipb[k];
    };

    // (loops over a thread's rings without branches: see march_fast_kernel)
    const bool dump_fields = mode == MODE_MARCH && W.dump_psi != nullptr;
    const int slice0 = slice;
    uint64_t t_start = 0;
    bool pending_push = false;  // the table arrays a, b, T, D, S hold the push of slice - 1
    bool blk_bad = false;   // this CTA failed the guard at slice - 1
    int far_skip = 0;       // (resort's memory of rings that moved far)
    int has_prev_before = has_prev;

    for (;;) {
        // the next slice's beam offsets, loaded here so that their latency
        // overlaps the exchange's cluster barrier
        int nxt0 = 0, nxt1 = 0;
        if (stg.cap > 0 && slice + 1 < s_end && slice + 1 < n_steps) {
            nxt0 = W.boff[slice + 1];
            nxt1 = W.boff[slice + 2];
        }
        // ---------------- exchange: order vote, edges, guard of the push
        {
            // time budget: thread 0 of the cluster's rank 0 decides for all
            // (flag 2 of the exchange); read after block_sorted's barrier
            if (W.budget_ns > 0 && crank == 0 && tid == 0) {
                const uint64_t now = global_ns();
                if (slice == slice0) t_start = now;
                s_stop = slice > slice0 && now - t_start >= (uint64_t)W.budget_ns;
            }
            // this slice's staged beam: wait (bounded) before the exchange,
            // so that a wait that gives up stops every CTA alike
            bool stalled = false;
            if (slice < s_end && (pending & (1 << (slice & 1)))) {
                const int bf = slice & 1;
                stalled = __syncthreads_or(!mbar_wait_bounded(&s_bar[bf], (parity >> bf) & 1u));
                parity ^= 1u << bf;
                pending &= ~(1 << bf);
            }
            const float* vr = pending_push ? sm.a : sm.rh;  // the state this slice would start from
            const bool srt = block_sorted<K>(vr, nl, p0);
            const bool stop = W.budget_ns > 0 && crank == 0 && s_stop;
            // flags: 1 failed the guard at slice - 1, 2 stop (time budget),
            // 4 this CTA's staging wait gave up
            if (tid < csize)
                *rmt(cl, &s_xch[crank], tid) = make_float4(srt ? 1.f : 0.f, vr[SW::at(0)], vr[SW::at(nl - 1)],
                                                           (blk_bad ? 1.f : 0.f) + (stop ? 2.f : 0.f) +
                                                               (stalled ? 4.f : 0.f));
        }
        cl.sync();
        bool any_bad = false, all_sorted = true, any_stalled = false;
        const bool stop_now = ((int)s_xch[0].w & 2) != 0;
        for (int r = 0; r < csize; ++r) {
            const float4 v = s_xch[r];
            const int fl = (int)v.w;
            if (fl & 1) any_bad = true;
            if (fl & 4) any_stalled = true;
            if (v.x == 0.f) all_sorted = false;
            if (r + 1 < csize && v.z > s_xch[r + 1].y) all_sorted = false;
        }
        if (any_bad) {  // slice - 1 failed the guard: its push is void
            status = 4;
            fail = slice - 1;
            has_prev = has_prev_before;
            break;
        }
        if (pending_push) {  // commit the push of slice - 1
#pragma unroll
            for (int k = 0; k < K; ++k) {
                int p = p0 + k;
                if (p < nl) {
                    const int a = SW::at(p);
                    sm.rh[a] = sm.a[a];
                    sm.rl[a] = sm.b[a];
                    sm.u[a] = sm.T[a];
                    sm.fr[a] = sm.D[a];
                    sm.fu[a] = sm.S[a];
                }
            }
            pending_push = false;
            __syncthreads();
        }
        if (any_stalled) {  // the wake stops before this slice
            status = WAKE_STATUS_TIMEOUT;
            fail = slice;
            break;
        }
        if (slice >= s_end || stop_now) break;
        // prefetch the next slice's beam while this one is solved (its
        // buffer was last read by slice - 1, before the last barrier)
        if (slice + 1 < s_end && stage_slice(stg, W, slice + 1, nxt0, nxt1 - nxt0, stall_armed)) {
            pending |= 1 << ((slice + 1) & 1);
            stall_armed = false;
        }
        const int sbuf = slice & 1;

        // ---------------- a2: sort by radius if out of order (cluster-wide)
        if (!all_sorted) {
            // local sort of every CTA's range, then every ring to its place
            resort<K>(sm, nl, far_skip);
            // (a NaN radius has no place: its CTA's edges tell, the rings stay,
            // and the guard stops the wake at this slice)
            bool nan = false;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (p0 + k < nl && isnan(sm.rh[SW::at(p0 + k)])) nan = true;
            nan = __syncthreads_or(nan);
            // every CTA's edges, pushed to all peers
            if (tid < csize) {
                const float none = __int_as_float(0x7fffffff);
                *rmt(cl, &s_edges[crank], tid) = nan ? make_float2(none, none)
                                                     : make_float2(sm.rh[SW::at(0)], sm.rh[SW::at(nl - 1)]);
            }
            cl.sync();
            bool move = false, all_numbers = true;
            for (int r = 0; r < csize; ++r) {
                if (isnan(s_edges[r].x)) all_numbers = false;
                if (r + 1 < csize && s_edges[r].y > s_edges[r + 1].x) move = true;
            }
            if (move && all_numbers) cluster_move<K>(cl, sm, n, TK, nl, scratch, s_edges, s_cnt, s_last);
            else if (tid < csize) s_last[tid] = s_edges[tid].y;
        } else if (tid < csize) {
            s_last[tid] = s_xch[tid].z;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int a = SW::at(p0 + k);
            const bool on = k < nv;
            rh[k] = on ? sm.rh[a] : 1.f;
            ur[k] = on ? sm.u[a] : 0.f;
            idv[k] = on ? sm.id[a] : 0;
            ir[k] = __frcp_rn(rh[k]);
        }

        // ---------------- a3: the beam's charge inside each ring
        int b0 = 0, m = 0;
        R qtot = 0;
        if (W.nb > 0 && slice < n_steps) {
            b0 = W.boff[slice];
            m = W.boff[slice + 1] - b0;
            qtot = W.bTot[slice];
        }
        // the slice's beam arrays: from this CTA's stage if they were staged
        SliceBeam sb = {W.br + b0, W.bQs + b0, W.bE + b0};
        const bool in_stage = stg.cap > 0 && stg.fits(m);
        if (in_stage)
            sb = {stg.arr(sbuf, 0) + (b0 & 3), stg.arr(sbuf, 1) + (b0 & 3), stg.arr(sbuf, 2) + (b0 & 3)};
        // The radii are searched in shared memory: in the stage, or, for a
        // slice that was not staged, in a copy in the dead region tables
        // where they fit them, else where they are.
        __syncthreads();  // (publishes s_last)
        const bool dist = m > T && csize > 1;
        {
            const bool copied = m > 0 && !in_stage && m <= kFastArrays / 2 * cap;
            SliceBeam sp = sb;
            if (copied) {  // into the dead tables a, b, T, D, S, psi
                float* prw = sm.a;
                for (int i0 = tid; i0 < m; i0 += kPartBatch * T) {
                    float v[kPartBatch];  // loads in flight together
#pragma unroll
                    for (int j = 0; j < kPartBatch; ++j) v[j] = i0 + j * T < m ? __ldg(W.br + b0 + i0 + j * T) : 0.f;
#pragma unroll
                    for (int j = 0; j < kPartBatch; ++j)
                        if (i0 + j * T < m) prw[i0 + j * T] = v[j];
                }
                __syncthreads();
                sp.br = prw;
            }
            ring_beam_field<K>(sp, m, qtot, inv_2pi_dxi, nv, rh, IR, bbv);
            if (copied) __syncthreads();  // the copy is overwritten from a5 on
        }

        // ---------------- a4: scan of (sum w, sum w ln rho)
        A sw = zeroA, sl = zeroA;
        R lp[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int a = SW::at(p0 + k);
            const bool on = k < nv;
            RingConst c = ring_const<K>(ctab, idv[k]);
            const R dl = ff_to_f(ff_acc(ff{rh[k], sm.rl[a]}, ff_neg(c.r0)));  // rho - rho0
            const R l1 = log1pf(dl * c.ir0);
            lp[k] = on ? l1 : 0.f;
            sw = ff_acc(sw, ff_if(on, c.w));
            sl = ff_acc(sl, ff_if(on, ff_acc(c.wl0, ff_two_prod(c.w.hi, l1))));
        }
        Pair<A> ex1;
        A Wtot, Ltot;
        {
            Pair<A> tot1, pre1, all1;
            // (one-barrier scans: a cluster barrier separates each from the next)
            ex1 = block_excl_scan1<false>(Pair<A>{sw, sl}, OpAddPair(), Pair<A>{zeroA, zeroA},
                                          reinterpret_cast<Pair<A>*>(sscan), tot1);
            cluster_push(cl, x1, tot1);
            cl.sync();
            fold_fwd_shared(x1, crank, csize, Pair<A>{zeroA, zeroA}, OpAddPair(), &f1[0], &f1[1]);
            pre1 = f1[0];
            all1 = f1[1];
            ex1 = OpAddPair()(pre1, ex1);
            Wtot = all1.x;
            Ltot = all1.y;
        }

        // ---------------- a5: psi, d_rho psi, psibar, gamma, t; the solve's matrices
        A S = ex1.x, L = ex1.y;
        A tl = zeroA;
        Mat2<R> Mf = I2, Mb = I2;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            int p = p0 + k;
            if (p < nl) {
                const int a = SW::at(p);
                RingConst c = ring_const<K>(ctab, idv[k]);
                R r = rh[k], u = ur[k];
                A rf = {r, sm.rl[a]};
                A r2 = ff_mul(rf, rf);
                A lnr = ff_add_f(c.ln0, lp[k]);
                A Ir = r < rmax ? ff_mul_f(r2, half_n) : Imax;
                A psion = r <= rmax ? ff_acc(c0, ff_neg(ff_mul_f(r2, quarter_n))) : ff_neg(ff_mul(Imax, lnr));
                R psi = ff_to_f(ff_acc(ff_acc(ff_acc(Ltot, ff_neg(L)), ff_mul(S, lnr)), psion));
                A Sm = ff_acc(S, ff_neg(Ir));
                R dpr = ff_to_f(ff_acc(Sm, c.wh)) * IR(k);
                R pb = 1.f + psi;
                R ip = __frcp_rn(pb);
                pbv[k] = pb;
                ipb[k] = ip;
                dprv[k] = dpr;
                tv[k] = c.w.hi * u * IR(k) * ip;
                sm.D[a] = ff_to_f(Sm);
                sm.S[a] = ff_to_f(S);
                sm.psi[a] = psi;
                {
                    const R wr = c.w.hi * IR(k), hA = 0.5f * (wr * ip);
                    hav[k] = hA;
                    Mat2<R> M = {1.f + hA * r, hA * IR(k), -hA * r * r * r, 1.f - hA * r};
                    Mf = OpMatLeft()(Mf, M);
                }
                if (K == 2 && mode == MODE_MARCH && W.dump_psi) {
                    size_t row = (size_t)slice * n + idv[k];
                    W.dump_psi[row] = psi;
                    W.dump_dpr[row] = dpr;
                }
                S = ff_acc(S, c.w);
                L = ff_acc(L, ff_acc(c.wl0, ff_two_prod(c.w.hi, lp[k])));
                tl = ff_add_f(tl, tv[k]);
            } else {
                pbv[k] = 1.f; ipb[k] = 1.f; dprv[k] = 0.f; tv[k] = 0.f; hav[k] = 0.f;
            }
        }
        if (K != 2 && dump_fields)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < nv) {
                    const size_t row = (size_t)slice * n + idv[k];
                    W.dump_psi[row] = sm.psi[SW::at(p0 + k)];
                    W.dump_dpr[row] = dprv[k];
                }
#pragma unroll
        for (int k = K - 1; k >= 0; --k) {
            R r = rh[k], hA = hav[k];
            Mat2<R> Mi = {1.f - hA * r, -hA * IR(k), hA * r * r * r, 1.f + hA * r};
            Mb = OpMatLeft()(Mb, Mi);
        }
        A Tex, Ttot;
        Mat2<R> Yf, Yb;
        {
            // this CTA's sum and its forward and reverse products go to every CTA
            A Ttot_blk;
            Mat2<R> tf, tb;
            Tex = block_excl_scan_sum_mats1<true>(tl, Mf, Mb, zeroA, reinterpret_cast<SumMats<A, R>*>(sscan), Yf, Yb,
                                                  Ttot_blk, tf, tb);
            if (tid < csize) {
                *rmt(cl, &x2[crank], tid) = Ttot_blk;
                *rmt(cl, &x3f[crank], tid) = tf;
                *rmt(cl, &x3r[crank], tid) = tb;
            }
            cl.sync();
            // the three folds by one thread each, of different warps where there are as many
            if (tid == 32 % T) {
                Mat2<R> pre, all;
                fold_rev(x3r, crank, csize, I2, OpMatLeft(), pre, all);
                f3[2] = pre;
            }
            if (tid == 64 % T) {
                A pre, all;
                fold_fwd(x2, crank, csize, zeroA, OpAdd(), pre, all);
                f2[0] = pre;
                f2[1] = all;
            }
            fold_fwd_shared(x3f, crank, csize, I2, OpMatLeft(), &f3[0], &f3[1]);
            Ttot = f2[1];
            Tex = ff_acc(f2[0], Tex);
            Yf = OpMatLeft()(f3[0], Yf);
            Yb = OpMatLeft()(f3[2], Yb);
        }

        // ---------------- a6 + a7
        {
            A Tacc = Tex;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                int p = p0 + k;
                if (p < nl) {
                    const int a = SW::at(p);
                    const float4* ct = ring_tab<K>(ctab, idv[k]);
                    const float4 cw = __ldg(ct + ctab.part);
                    const R w = cw.x, wh = cw.z;
                    R r = rh[k], u = ur[k], dpr = dprv[k], ip = IPB(k), iR = IR(k);
                    sm.T[a] = ff_to_f(ff_acc(Ttot, ff_neg(Tacc)));
                    Tacc = ff_add_f(Tacc, tv[k]);
                    R above = ff_to_f(ff_acc(Ttot, ff_neg(Tacc)));
                    R dpz = -(above + (1.f - wh * __ldg(reinterpret_cast<const float*>(ct + 2 * ctab.part) + 2)) * tv[k]);
                    tv[k] = dpz;
                    R pb = pbv[k];
                    R g = 0.5f * (1.f + u * u + pb * pb) * ip;
                    R wr = w * iR, ip2 = ip * ip, uu = u * u;
                    R Ac = wr * ip;
                    R Bc = wr * ip2 * (-g * dpr + bbv[k] * pb + uu * dpr * ip - u * dpz) + wr * iR * uu * ip2;
                    R Cc = -wr * (g * ip - 1.f - uu * ip2);
                    s0v[k] = 0.25f * (2.f * Bc + Ac * Cc);
                    s1v[k] = 0.25f * r * (4.f * Cc - 2.f * Bc * r - Ac * Cc * r);
                    if (K == 2 && mode == MODE_MARCH && W.dump_dpz) W.dump_dpz[(size_t)slice * n + idv[k]] = dpz;
                } else {
                    s0v[k] = 0.f; s1v[k] = 0.f;
                }
            }
            if (K != 2 && dump_fields)
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < nv) W.dump_dpz[(size_t)slice * n + idv[k]] = tv[k];
        }

        // ---------------- a8: B_theta^(p)
        R Rra[K], Rrb[K], Dda[K], Ddb[K];
        {
            Mat2<R> Y = Yf;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                R r = rh[k], hA = hav[k];
                Mat2<R> M = {1.f + hA * r, hA * IR(k), -hA * r * r * r, 1.f - hA * r};
                Y = OpMatLeft()(Y, M);
                Rra[k] = Y.m00;
                Rrb[k] = Y.m10;
            }
        }
        A gl = zeroA, dl = zeroA;
        R gpv[K], dpv[K];
        R Dp0a, Dp0b;
        {
            Mat2<R> Y = Yb;
#pragma unroll
            for (int k = K - 1; k >= 0; --k) {
                Dda[k] = Y.m01;
                Ddb[k] = Y.m11;
                gpv[k] = 0.f;
                dpv[k] = 0.f;
                if (p0 + k < nl) {
                    R q0 = Rra[k], q1 = Rrb[k], d0 = Y.m01, d1 = Y.m11;
                    R iw = __frcp_rn(q0 * d1 - q1 * d0);
                    R gp = (s0v[k] * d1 - s1v[k] * d0) * iw;
                    R dp = (q0 * s1v[k] - q1 * s0v[k]) * iw;
                    gpv[k] = gp;
                    dpv[k] = dp;
                    gl = ff_add_f(gl, gp);
                    dl = ff_add_f(dl, dp);
                    R r = rh[k], hA = hav[k];
                    Mat2<R> Mi = {1.f - hA * r, -hA * IR(k), hA * r * r * r, 1.f + hA * r};
                    Y = OpMatLeft()(Y, Mi);
                }
            }
            Dp0a = Y.m01;
            Dp0b = Y.m11;
        }
        A g_tot, d_tot;
        Pair<A> gd = block_excl_scan_fwd_rev1(dl, gl, zeroA, reinterpret_cast<Pair<A>*>(sscan), d_tot, g_tot);
        A all4f;
        {
            if (tid < csize) {
                *rmt(cl, &x4f[crank], tid) = d_tot;
                *rmt(cl, &x4r[crank], tid) = g_tot;
            }
            cl.sync();
            if (tid == 32 % T) {
                A pre, all;
                fold_rev(x4r, crank, csize, zeroA, OpAdd(), pre, all);
                f4[2] = pre;
            }
            fold_fwd_shared(x4f, crank, csize, zeroA, OpAdd(), &f4[0], &f4[1]);
            all4f = f4[1];
            gd.x = ff_acc(f4[0], gd.x);
            gd.y = ff_acc(f4[2], gd.y);
        }
        {
            R Gk[K];
            A Gsuf = gd.y;
#pragma unroll
            for (int k = K - 1; k >= 0; --k) {
                Gsuf = ff_add_f(Gsuf, gpv[k]);
                Gk[k] = ff_to_f(Gsuf);
            }
            A Hex = gd.x;
            R Rpa = Yf.m00, Rpb = Yf.m10;
            R Dpa = Dp0a, Dpb = Dp0b;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                int p = p0 + k;
                if (p < nl) {
                    R G = Gk[k];
                    R H = ff_to_f(Hex);
                    int a = SW::at(p);
                    sm.a[a] = -G * Rpa + H * Dpa;
                    sm.b[a] = -G * Rpb + H * Dpb;
                    Hex = ff_add_f(Hex, dpv[k]);
                    Rpa = Rra[k];
                    Rpb = Rrb[k];
                    Dpa = Dda[k];
                    Dpb = Ddb[k];
                }
            }
            if (last_cta && p0 < nl && p0 + K >= nl) {  // region n
                const int a = nl < TK ? SW::at(nl) : TK;
                sm.a[a] = 0.f;
                sm.b[a] = ff_to_f(all4f);
                sm.T[a] = 0.f;
                sm.D[a] = ff_to_f(ff_acc(Wtot, ff_neg(Imax)));
                sm.S[a] = ff_to_f(Wtot);
                sm.psi[a] = 0.f;
            }
        }
        // the next CTA's first region, for B^(p) at this CTA's last ring
        if (tid == 0 && crank > 0) *rmt(cl, &s_nab, crank - 1) = make_float2(sm.a[SW::at(0)], sm.b[SW::at(0)]);
        cl.sync();

        // ---------------- B^(p) at the rings and the guard
        bool bad = false;
        R bpv[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int p = p0 + k, a = SW::at(p);
            const bool on = k < nv;
            // the next region: the next ring's, region n, or the next CTA's first
            const bool in = p + 1 < nl;
            const int a1 = in ? SW::at(p + 1) : nl < TK ? SW::at(nl) : TK;
            const R a1v = in || last_cta ? sm.a[a1] : s_nab.x, b1v = in || last_cta ? sm.b[a1] : s_nab.y;
            const R bp = 0.5f * ((sm.a[a] + a1v) * rh[k] + (sm.b[a] + b1v) * IR(k));
            bpv[k] = on ? bp : 0.f;
            const R pb = pbv[k];
            bad = bad || (on && (!(pb > 0.f) || !isfinite(pb) || !isfinite(dprv[k]) || !isfinite(tv[k]) ||
                                 !isfinite(bp) || !isfinite(bbv[k])));
        }
        if (mode == MODE_MARCH && W.dump_r)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < nv) {
                    const size_t row = (size_t)slice * n + idv[k];
                    W.dump_r[row] = rh[k];
                    if (W.dump_ur) {
                        W.dump_ur[row] = ur[k];
                        W.dump_bp[row] = bpv[k];
                        W.dump_bb[row] = bbv[k];
                    }
                }

        // ---------------- a9: fields on the beam particles (or query radii)
        // Region k (radii in (rho_{k-1}, rho_k]) lives in the CTA holding
        // ring k, region n in the last CTA: this CTA serves the radii in
        // (previous CTA's last radius, its own last radius].
        {
            const float lo_r = crank > 0 ? s_last[crank - 1] : -INFINITY;
            const float hi_r = last_cta ? INFINITY : s_last[crank];
            if (mode == MODE_MARCH) {
                // the particles of this CTA's own range, or (more of them than
                // threads) an even share of the slice with the owner's
                // tables read remotely; region k (radii in (rho_{k-1}, rho_k]) lives in the CTA
                // holding ring k, region n in the last CTA
                const int mc = dist ? (m + csize - 1) / csize : m;
                const int c0q = dist ? crank * mc : 0;
                const int c1q = dist ? min(m, c0q + mc) : m;
                const int per = (c1q - c0q + T - 1) / T;
                const int q0 = c0q + tid * per, q1 = min(c1q, q0 + per);
                int o = crank, kr = -1;  // owner of the current run and its tables (kr -1: no rank in them yet)
                FastSmem so = sm;
                int nl_o = nl;
                bool past = false;
                for (int qb = q0; qb < q1 && !past; qb += kPartBatch) {
                  float xb[kPartBatch], qb_s[kPartBatch];  // loaded together, then evaluated
#pragma unroll
                  for (int j = 0; j < kPartBatch; ++j) {
                      xb[j] = qb + j < q1 ? sb.br[qb + j] : INFINITY;
                      qb_s[j] = qb + j < q1 ? sb.qs[qb + j] : 0.f;
                  }
#pragma unroll
                  for (int j = 0; j < kPartBatch; ++j) {
                    const int q = qb + j;
                    const R x = xb[j];
                    if (q >= q1) {
                        past = true;
                        break;
                    }
                    if (!dist && !(x > lo_r)) continue;
                    int o2 = dist && q == q0 ? 0 : o;  // owners only grow along the run
                    while (o2 + 1 < csize && !(x <= s_last[o2])) ++o2;
                    if (!dist && o2 != crank) {
                        past = true;
                        break;
                    }
                    if (o2 != o) {
                        o = o2;
                        so = o == crank ? sm : rmt_sm(cl, sm, o);
                        nl_o = min(TK, n - o * TK);
                        kr = -1;
                    }
                    R psi, dpr, dpz, bp, bb = 0.f;
                    if (x > 0.f) {
                        kr = kr < 0 ? ring_rank_all<K>(so.rh, nl_o, x) : ring_rank_from<K>(so.rh, nl_o, kr, x);
                        fast_fields_region<K>(so, nl_o, TK, kr, x, rmax, half_n, quarter_n, Wtot, Imax, c0, &dpr,
                                              &dpz, &bp, &psi);
                        bb = qb_s[j] * inv_2pi_dxi / x;
                    } else {
                        psi = ff_to_f(ff_add(Ltot, c0));
                        dpr = 0.f;
                        dpz = -ff_to_f(Ttot);
                        bp = 0.f;
                    }
                    const int64_t o_idx = b0 + q;
                    W.out_ez[o_idx] = -dpz;
                    W.out_wr[o_idx] = -dpr;
                    W.out_bt[o_idx] = bp + bb;
                    W.out_psi[o_idx] = psi;
                  }
                }
                // no CTA may overwrite its tables (the push lands there)
                // while another still reads them
                if (dist) cl.sync();
            } else {
                const int64_t q_step = (int64_t)(gridDim.x / csize) * T;
                for (int64_t q = (int64_t)widx * T + tid; q < W.nq; q += q_step) {
                    const R x = (R)W.rq[q];
                    // a radius belongs here if lo_r < x <= hi_r (CTA 0 also
                    // takes a NaN query, which no comparison places)
                    if (!(x > lo_r && x <= hi_r) && !(crank == 0 && x != x)) continue;
                    R psi, dpr, dpz, bp, bb = 0.f;
                    if (x > 0.f) {
                        const int kl = ring_rank<K>(sm.rh, nl, x);
                        fast_fields_region<K>(sm, nl, TK, kl, x, rmax, half_n, quarter_n, Wtot, Imax, c0, &dpr,
                                              &dpz, &bp, &psi);
                        if (m > 0) {
                            int l2 = lower_bound_dev(W.br + b0, m, x);
                            R Q = l2 < m ? W.bE[b0 + l2] : qtot;
                            bb = Q * inv_2pi_dxi / x;
                        }
                    } else {
                        psi = ff_to_f(ff_add(Ltot, c0));
                        dpr = 0.f;
                        dpz = -ff_to_f(Ttot);
                        bp = 0.f;
                    }
                    if (W.q_ez) W.q_ez[q] = -dpz;
                    if (W.q_wr) W.q_wr[q] = -dpr;
                    if (W.q_bt) W.q_bt[q] = bp + bb;
                    if (W.q_psi) W.q_psi[q] = psi;
                }
            }
        }
        blk_bad = __syncthreads_or(bad);  // (every read of the tables is done)
        if (mode != MODE_MARCH) break;

        // ---------------- a10: AB2 push into the table arrays (dead after
        // a9); it becomes the state at the next exchange unless some CTA
        // failed the guard
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int a = SW::at(p0 + k);
            R u = ur[k], pb = pbv[k], ip = IPB(k);
            R g = 0.5f * (1.f + u * u + pb * pb) * ip;
            R fr = u * ip;
            R fu = g * dprv[k] * ip - (bpv[k] + bbv[k]);
            const R drr = dxi * (has_prev ? 1.5f * fr - 0.5f * sm.fr[a] : fr);
            const R du = dxi * (has_prev ? 1.5f * fu - 0.5f * sm.fu[a] : fu);
            ff rr = ff_add_f(ff{rh[k], sm.rl[a]}, drr);
            R un = u + du;
            const bool over = rr.hi < 0.f;  // through the axis: the ring reappears at -rho
            rr = over ? ff_neg(rr) : rr;
            un = over ? -un : un;
            fr = over ? -fr : fr;
            fu = over ? -fu : fu;
            if (k < nv) {
                sm.a[a] = rr.hi;
                sm.b[a] = rr.lo;
                sm.T[a] = un;
                sm.D[a] = fr;
                sm.S[a] = fu;
            }
        }
        has_prev_before = has_prev;
        has_prev = 1;
        pending_push = true;
        ++slice;
        __syncthreads();  // the pushed state is read across threads next
    }
    // no bulk copy may still write this CTA's shared memory when it exits:
    // wait (bounded) for any staged slice that was not consumed
    for (int bf = 0; bf < 2; ++bf)
        if ((pending & (1 << bf)) && !mbar_wait_bounded(&s_bar[bf], (parity >> bf) & 1u) && status == 0) {
            status = WAKE_STATUS_TIMEOUT;
            fail = slice;
        }
    cl.sync();  // no CTA leaves while a peer may still touch its shared memory
    if (mode == MODE_QUERY) return;  // (the state stays as the march left it: other clusters may still load it)

    for (int p = tid; p < nl; p += T) {
        int a = SW::at(p), g = base + p;
        W.rho[buf][g] = sm.rh[a];
        W.rho_lo[g] = sm.rl[a];
        W.ur[buf][g] = sm.u[a];
        W.frho[buf][g] = sm.fr[a];
        W.fur[buf][g] = sm.fu[a];
        W.rid[buf][g] = sm.id[a];
    }
    if (tid == 0 && crank == 0) {
        put_march_times(W.ctl, t_launch);
        W.ctl[CTL_NEXT] = slice;
        W.ctl[CTL_PREV] = has_prev;
        if (status) {
            W.ctl[CTL_STATUS] = status;
            W.ctl[CTL_FAIL] = fail;
        }
    }
}

}  // namespace gbwake
