// rank_sort.cuh -- where each ring of a nearly sorted list goes: a stable
// rank by counting, in place of a sorting network.
//
// Between two slices rings move by a few places, so the sorted place of ring
// p is p less the earlier rings above it plus the later rings below it.
// Running maxima from the front and minima from the back over chunks of 8
// tell where that count can stop, and the chunks' own extremes which chunks
// hold nothing to count: two reads for a chunk that is skipped, eight for
// one that is counted.  O(n) to prepare, then every ring's rank by itself:
// two barriers, where the bitonic network takes log2(n)^2 / 2 with one
// barrier each and one block of the cluster working (measured on GB300 with
// the two-species, RK4 and beam-grid marches; times at their kernels).  A
// list out of order over long distances only costs time: the count runs on.
//
// Keys are the radii's bit patterns as signed integers, which order as the
// radii do (they are >= 0) and give a total order whatever they hold, so the
// ranks are a permutation; equal keys keep their order (the stable sort).
#pragma once

#include "common.cuh"

namespace gbwake {

__device__ __forceinline__ int32_t radius_key(float r) { return __float_as_int(r); }
__device__ __forceinline__ int64_t radius_key(double r) { return __double_as_longlong(r); }

struct OpMax {
    template <class T>
    __device__ __forceinline__ T operator()(T a, T b) const { return a < b ? b : a; }
};
struct OpMin {
    template <class T>
    __device__ __forceinline__ T operator()(T a, T b) const { return b < a ? b : a; }
};

template <class R>
struct RankSort {
    using KT = decltype(radius_key(R()));
    static constexpr int kChunk = 8;
    static constexpr KT kLow = (KT)((uint64_t)1 << (8 * sizeof(KT) - 1));
    static constexpr KT kHigh = (KT)~kLow;
    const R* r;            // [n] radii, block-visible
    KT *cmax, *cmin;       // [chunks] the chunks' extremes
    KT *pmax, *smin;       // [chunks] maxima of the chunks up to, minima of the chunks from
    int n;

    __host__ __device__ static int chunks(int n) { return (n + kChunk - 1) / kChunk; }
    __host__ __device__ static size_t bytes(int n) { return (size_t)4 * chunks(n) * sizeof(KT); }
    // `mem`: bytes(n) of shared memory
    __device__ __forceinline__ RankSort(const R* radii, int n_, void* mem) : r(radii), n(n_) {
        const int c = chunks(n);
        cmax = static_cast<KT*>(mem);
        cmin = cmax + c;
        pmax = cmin + c;
        smin = pmax + c;
    }
    // Every thread of the block; the radii are visible to it already.  scan:
    // 2 x 32 keys of shared memory.  Ends with a barrier.
    __device__ void prepare(KT* scan) {
        const int c = chunks(n), T = blockDim.x, tid = threadIdx.x;
        const int per = (c + T - 1) / T, c0 = min(c, tid * per), c1 = min(c, c0 + per);
        KT mx = kLow, mn = kHigh;
        for (int i = c0; i < c1; ++i) {
            KT a = kLow, b = kHigh;
            for (int q = i * kChunk; q < min(n, (i + 1) * kChunk); ++q) {
                const KT v = radius_key(r[q]);
                a = OpMax()(a, v);
                b = OpMin()(b, v);
            }
            cmax[i] = a;
            cmin[i] = b;
            mx = OpMax()(mx, a);
            mn = OpMin()(mn, b);
        }
        KT tot;
        KT pre = block_excl_scan1<false>(mx, OpMax(), kLow, scan, tot);
        KT suf = block_excl_scan1<true>(mn, OpMin(), kHigh, scan + 32, tot);
        for (int i = c0; i < c1; ++i) pmax[i] = pre = OpMax()(pre, cmax[i]);
        for (int i = c1 - 1; i >= c0; --i) smin[i] = suf = OpMin()(suf, cmin[i]);
        __syncthreads();
    }
    // the sorted place of ring p (its radius x)
    __device__ int place(int p, R radius) const {
        const KT x = radius_key(radius);
        const int c = p / kChunk, nc = chunks(n);
        int at = p;
        for (int q = c * kChunk; q < p; ++q) at -= radius_key(r[q]) > x;
        for (int q = p + 1; q < min(n, (c + 1) * kChunk); ++q) at += radius_key(r[q]) < x;
        for (int i = c - 1; i >= 0 && pmax[i] > x; --i)
            if (cmax[i] > x)
#pragma unroll
                for (int q = 0; q < kChunk; ++q) at -= radius_key(r[i * kChunk + q]) > x;
        for (int i = c + 1; i < nc && smin[i] < x; ++i)
            if (cmin[i] < x)
                for (int q = i * kChunk; q < min(n, (i + 1) * kChunk); ++q) at += radius_key(r[q]) < x;
        return at;
    }
};

}  // namespace gbwake
