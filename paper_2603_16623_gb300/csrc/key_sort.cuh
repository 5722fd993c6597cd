// key_sort.cuh -- the per-thread steps of the on-chip re-sort (march_fast.cuh):
// (key, previous position) pairs in the order of the stable sort, sorted in
// registers, split against a neighbour's run, merged pairwise.
//
// Keys are the radii's bit patterns as signed integers: radii are >= 0, so
// these order as the radii do, and unlike a comparison of floats they order
// whatever a radius holds -- a push from a non-finite or overflowing history
// leaves a NaN, which sorts beyond every number and stays in its ring, so that
// the places are a permutation of the rings and the slice's guard finds it.
// With an order that a NaN leaves undecided a merge may take more entries of
// one run than there are.  Compiles for the host too (tests).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define WK_HD __host__ __device__ __forceinline__
#define WK_UNROLL _Pragma("unroll")
#else
#define WK_HD inline
#define WK_UNROLL
#endif

namespace gbwake {

struct KeySrc {
    int32_t key;
    int32_t src;
};
// the key of a position without a ring: with its position (beyond every
// ring's) it sorts after all rings
constexpr int32_t kNoRingKey = 0x7fffffff;

WK_HD bool ks_less(const KeySrc& a, const KeySrc& b) { return a.key < b.key || (a.key == b.key && a.src < b.src); }
WK_HD void ks_order(KeySrc& a, KeySrc& b) {
    if (ks_less(b, a)) {
        KeySrc t = a;
        a = b;
        b = t;
    }
}
// sorts v[0, K) ascending (K a power of two): bitonic network, static indices
template <int K>
WK_HD void ks_sort(KeySrc (&v)[K]) {
    WK_UNROLL
    for (int k2 = 2; k2 <= K; k2 <<= 1)
        WK_UNROLL
        for (int j = k2 >> 1; j > 0; j >>= 1)
            WK_UNROLL
            for (int i = 0; i < K; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    if ((i & k2) == 0) ks_order(v[i], v[l]);
                    else ks_order(v[l], v[i]);
                }
            }
}
// a bitonic v (after a half-cleaner) into ascending order
template <int K>
WK_HD void ks_bitonic_finish(KeySrc (&v)[K]) {
    WK_UNROLL
    for (int j = K >> 1; j > 0; j >>= 1)
        WK_UNROLL
        for (int i = 0; i < K; ++i) {
            const int l = i ^ j;
            if (l > i) ks_order(v[i], v[l]);
        }
}
// v and a neighbour's run (at(k): its k-th entry), both ascending: the lower
// half of both (left) or the upper, ascending
template <int K, class At>
WK_HD void ks_merge_split(KeySrc (&v)[K], At at, bool left) {
    WK_UNROLL
    for (int k = 0; k < K; ++k) {  // half-cleaner against the run, reversed
        const KeySrc w = at(K - 1 - k);
        const bool lt = ks_less(v[k], w);
        if (left ? !lt : lt) v[k] = w;
    }
    ks_bitonic_finish<K>(v);
}
// Outputs [d, d + K) of the merge of the ascending runs at(0 .. nA) and
// at(L .. L + nB) (d + K <= nA + nB): put(k, entry).  A run's end is told by
// its index, so that no index leaves the two runs whatever the keys are.
template <int K, class At, class Put>
WK_HD void ks_merge_outputs(At at, int L, int nA, int nB, int d, Put put) {
    int lo = d > nB ? d - nB : 0, hi = d < nA ? d : nA;
    while (lo < hi) {  // outputs before d taken from the first run
        const int mid = (lo + hi) >> 1;
        if (ks_less(at(L + d - 1 - mid), at(mid))) hi = mid;
        else lo = mid + 1;
    }
    int i = lo, j = d - lo;
    KeySrc x = {kNoRingKey, 0}, y = x;
    if (i < nA) x = at(i);
    if (j < nB) y = at(L + j);
    WK_UNROLL
    for (int k = 0; k < K; ++k) {
        const bool take = j >= nB || (i < nA && !ks_less(y, x));
        put(k, take ? x : y);
        if (k + 1 < K) {
            if (take) {
                if (++i < nA) x = at(i);
            } else {
                if (++j < nB) y = at(L + j);
            }
        }
    }
}

}  // namespace gbwake
