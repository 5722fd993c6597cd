// common.cuh -- device utilities of the wake solver: float-float arithmetic,
// the two precision policies, and block-wide scans for associative (not
// necessarily commutative) operators in either direction.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ring_jump.cuh"  // (Mat2)

namespace gbwake {

// control words of a wake (device ints): next slice, status, failing
// slice, ring-state buffer, AB2 history present; CTL_T_BEGIN and CTL_T_END
// (two words each) the device time (globaltimer ns) at which the last march
// launch began and finished marching the wake
enum { CTL_NEXT = 0, CTL_STATUS = 1, CTL_FAIL = 2, CTL_BUF = 3, CTL_PREV = 4, CTL_T_BEGIN = 8, CTL_T_END = 10,
       CTL_N = 16 };
// the wake status codes the kernels write into CTL_STATUS (the values of
// include/wake.h's WAKE_EINVAL, WAKE_ENONFINITE, WAKE_ETIMEOUT)
enum { WAKE_STATUS_INVALID = 1, WAKE_STATUS_NONFINITE = 4, WAKE_STATUS_TIMEOUT = 5 };

// ---------------------------------------------------------------------------
// float-float ("ff"): an unevaluated sum hi + lo of two floats (~48-bit
// significand).  Knuth's TwoSum and the FMA-based exact product; nothing here
// multiplies and adds in one expression except through fmaf.
// ---------------------------------------------------------------------------
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b) {
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ ff ff_fast_two_sum(float a, float b) {  // |a| >= |b|
    float s = __fadd_rn(a, b);
    float e = __fsub_rn(b, __fsub_rn(s, a));
    return {s, e};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    ff s = ff_two_sum(a.hi, b.hi);
    ff t = ff_two_sum(a.lo, b.lo);
    s.lo = __fadd_rn(s.lo, t.hi);
    s = ff_fast_two_sum(s.hi, s.lo);
    s.lo = __fadd_rn(s.lo, t.lo);
    return ff_fast_two_sum(s.hi, s.lo);
}
// Accumulation add ("sloppy" float-float add): the error stays ~2^-46 of
// |a| + |b|; used where a running sum meets one more term.
__device__ __forceinline__ ff ff_acc(ff a, ff b) {
    ff s = ff_two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return ff_fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ ff ff_if(bool on, ff a) { return {on ? a.hi : 0.f, on ? a.lo : 0.f}; }
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ ff ff_add_f(ff a, float b) {
    ff s = ff_two_sum(a.hi, b);
    s.lo = __fadd_rn(s.lo, a.lo);
    return ff_fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ ff ff_two_prod(float a, float b) {
    float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return ff_fast_two_sum(p, e);
}
__device__ __forceinline__ ff ff_mul_f(ff a, float b) {
    float p = __fmul_rn(a.hi, b);
    float e = fmaf(a.hi, b, -p);
    e = fmaf(a.lo, b, e);
    return ff_fast_two_sum(p, e);
}
__device__ __forceinline__ float ff_to_f(ff a) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ ff ff_from_d(double d) {
    float h = (float)d;
    return {h, (float)(d - (double)h)};
}

// ---------------------------------------------------------------------------
// precision policies
//   PrecF64   : everything in double (the plain path)
//   PrecMixed : state, pushes and field evaluation in float; radial prefix
//               sums, psi and d_rho psi assembled in float-float
// ---------------------------------------------------------------------------
struct PrecF64 {
    using R = double;
    using A = double;
};
struct PrecMixed {
    using R = float;
    using A = ff;
};

// accumulator helpers, overloaded on the accumulator type
__device__ __forceinline__ double acc_zero(double) { return 0.0; }
__device__ __forceinline__ ff acc_zero(ff) { return {0.f, 0.f}; }
__device__ __forceinline__ double acc_add(double a, double b) { return a + b; }
__device__ __forceinline__ int64_t acc_add(int64_t a, int64_t b) { return a + b; }
// accumulations and scans of float-float values use the accumulation add
// (its error stays ~2^-46 of the operands' magnitudes)
__device__ __forceinline__ ff acc_add(ff a, ff b) { return ff_acc(a, b); }
__device__ __forceinline__ double acc_sub(double a, double b) { return a - b; }
__device__ __forceinline__ ff acc_sub(ff a, ff b) { return ff_sub(a, b); }
__device__ __forceinline__ double acc_add_r(double a, double b) { return a + b; }
__device__ __forceinline__ ff acc_add_r(ff a, float b) { return ff_add_f(a, b); }
__device__ __forceinline__ double acc_mul_r(double a, double b) { return a * b; }
__device__ __forceinline__ ff acc_mul_r(ff a, float b) { return ff_mul_f(a, b); }
__device__ __forceinline__ double acc_to_r(double a) { return a; }
__device__ __forceinline__ float acc_to_r(ff a) { return ff_to_f(a); }
__device__ __forceinline__ double acc_from_d(double d, double) { return d; }
__device__ __forceinline__ ff acc_from_d(double d, ff) { return ff_from_d(d); }
// exact square of a real as an accumulator
__device__ __forceinline__ double acc_sq(double x) { return x * x; }
__device__ __forceinline__ ff acc_sq(float x) { return ff_two_prod(x, x); }

__device__ __forceinline__ double real_log(double x) { return log(x); }
__device__ __forceinline__ float real_log(float x) { return logf(x); }
__device__ __forceinline__ bool real_finite(double x) { return isfinite(x); }
__device__ __forceinline__ bool real_finite(float x) { return isfinite(x); }

// ---------------------------------------------------------------------------
// shuffles for the scanned types
// ---------------------------------------------------------------------------
__device__ __forceinline__ double shfl_up_t(double v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double shfl_dn_t(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ int64_t shfl_up_t(int64_t v, int o) {
    return (int64_t)__shfl_up_sync(0xffffffffu, (long long)v, o);
}
__device__ __forceinline__ int64_t shfl_dn_t(int64_t v, int o) {
    return (int64_t)__shfl_down_sync(0xffffffffu, (long long)v, o);
}
__device__ __forceinline__ int32_t shfl_up_t(int32_t v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ int32_t shfl_dn_t(int32_t v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ int32_t shfl_idx_t(int32_t v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ float shfl_up_t(float v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float shfl_dn_t(float v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ ff shfl_up_t(ff v, int o) { return {shfl_up_t(v.hi, o), shfl_up_t(v.lo, o)}; }
__device__ __forceinline__ ff shfl_dn_t(ff v, int o) { return {shfl_dn_t(v.hi, o), shfl_dn_t(v.lo, o)}; }
__device__ __forceinline__ double shfl_idx_t(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ float shfl_idx_t(float v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ int64_t shfl_idx_t(int64_t v, int l) {
    return (int64_t)__shfl_sync(0xffffffffu, (long long)v, l);
}
__device__ __forceinline__ ff shfl_idx_t(ff v, int l) { return {shfl_idx_t(v.hi, l), shfl_idx_t(v.lo, l)}; }

template <class T>
struct Pair {
    T x, y;
};
template <class T>
__device__ __forceinline__ Pair<T> shfl_up_t(Pair<T> v, int o) { return {shfl_up_t(v.x, o), shfl_up_t(v.y, o)}; }
template <class T>
__device__ __forceinline__ Pair<T> shfl_dn_t(Pair<T> v, int o) { return {shfl_dn_t(v.x, o), shfl_dn_t(v.y, o)}; }
template <class T>
__device__ __forceinline__ Pair<T> shfl_idx_t(Pair<T> v, int l) { return {shfl_idx_t(v.x, l), shfl_idx_t(v.y, l)}; }

template <class R>
__device__ __forceinline__ Mat2<R> shfl_up_t(Mat2<R> v, int o) {
    return {shfl_up_t(v.m00, o), shfl_up_t(v.m01, o), shfl_up_t(v.m10, o), shfl_up_t(v.m11, o)};
}
template <class R>
__device__ __forceinline__ Mat2<R> shfl_dn_t(Mat2<R> v, int o) {
    return {shfl_dn_t(v.m00, o), shfl_dn_t(v.m01, o), shfl_dn_t(v.m10, o), shfl_dn_t(v.m11, o)};
}
template <class R>
__device__ __forceinline__ Mat2<R> shfl_idx_t(Mat2<R> v, int l) {
    return {shfl_idx_t(v.m00, l), shfl_idx_t(v.m01, l), shfl_idx_t(v.m10, l), shfl_idx_t(v.m11, l)};
}
// ---------------------------------------------------------------------------
// operators: op(a, b) = "a, then b" where a covers the earlier elements of
// the scan order
// ---------------------------------------------------------------------------
struct OpAdd {
    template <class T>
    __device__ __forceinline__ T operator()(T a, T b) const { return acc_add(a, b); }
};
struct OpAddPair {
    template <class T>
    __device__ __forceinline__ Pair<T> operator()(Pair<T> a, Pair<T> b) const {
        return {acc_add(a.x, b.x), acc_add(a.y, b.y)};
    }
};
// matrix product, later element on the left: result = b * a
struct OpMatLeft {
    template <class R>
    __device__ __forceinline__ Mat2<R> operator()(Mat2<R> a, Mat2<R> b) const {
        return {b.m00 * a.m00 + b.m01 * a.m10, b.m00 * a.m01 + b.m01 * a.m11,
                b.m10 * a.m00 + b.m11 * a.m10, b.m10 * a.m01 + b.m11 * a.m11};
    }
    static constexpr bool kDev = false;  // (operands as they are: see OpMatDevLeft)
    template <class R>
    __device__ __forceinline__ static Mat2<R> one() { return {1, 0, 0, 1}; }
    template <class R>
    __device__ __forceinline__ static Mat2<R> whole(Mat2<R> m) { return m; }
};
// ---------------------------------------------------------------------------
// block-wide exclusive scan.  REV = false: thread order 0, 1, ...;
// REV = true: the scan runs from the last thread down.  blockDim.x must be a
// multiple of 32 (<= 1024).  sbuf must hold 33 values of T in shared memory.
// Returns the exclusive fold of the earlier threads' values; `total` gets the
// fold over the whole block.  Contains barriers: every thread must call.
// ---------------------------------------------------------------------------
template <bool REV, class T, class Op>
__device__ __forceinline__ T warp_incl_scan(T v, Op op) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        T o = REV ? shfl_dn_t(v, off) : shfl_up_t(v, off);
        bool take = REV ? (lane + off < 32) : (lane >= off);
        if (take) v = op(o, v);
    }
    return v;
}

// the same over lanes [0, n) only, the others holding the identity: the
// steps of n lanes give bitwise what all five would
template <bool REV, class T, class Op>
__device__ __forceinline__ T warp_incl_scan_n(T v, Op op, int n) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        if (off >= n) break;
        T o = REV ? shfl_dn_t(v, off) : shfl_up_t(v, off);
        bool take = REV ? (lane + off < 32) : (lane >= off);
        if (take) v = op(o, v);
    }
    return v;
}
// the lane that holds the fold of lanes [0, n) after warp_incl_scan_n (in
// the association that the full scan leaves in lane 31)
__device__ __forceinline__ int scan_last_lane(int n) { return n > 1 ? (1 << (32 - __clz(n - 1))) - 1 : 0; }

template <bool REV, class T, class Op>
__device__ T block_excl_scan(T v, Op op, T ident, T* sbuf, T& total) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T inc = warp_incl_scan<REV>(v, op);
    T lex = REV ? shfl_dn_t(inc, 1) : shfl_up_t(inc, 1);
    if (REV ? (lane == 31) : (lane == 0)) lex = ident;
    if (REV ? (lane == 0) : (lane == 31)) sbuf[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T wv = lane < nw ? sbuf[lane] : ident;
        T winc = warp_incl_scan<REV>(wv, op);
        T wex = REV ? shfl_dn_t(winc, 1) : shfl_up_t(winc, 1);
        if (REV ? (lane == 31) : (lane == 0)) wex = ident;
        __syncwarp();
        if (lane < nw) sbuf[lane] = wex;
        if (lane == (REV ? 0 : 31)) sbuf[32] = winc;
    }
    __syncthreads();
    T res = op(sbuf[warp], lex);
    total = sbuf[32];
    __syncthreads();
    return res;
}

// One pass of two sums in opposite directions: fx scanned from thread 0 up,
// ry from the last thread down (same barriers as one scan).  Returns the
// exclusive forward sum of fx and the exclusive reverse (suffix) sum of ry;
// totals in tx, ty.  sbuf holds 33 Pair<T>.
template <class T>
__device__ Pair<T> block_excl_scan_fwd_rev(T fx, T ry, T zero, Pair<T>* sbuf, T& tx, T& ty) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T ix = warp_incl_scan<false>(fx, OpAdd());
    T iy = warp_incl_scan<true>(ry, OpAdd());
    T ex = shfl_up_t(ix, 1), ey = shfl_dn_t(iy, 1);
    if (lane == 0) ex = zero;
    if (lane == 31) ey = zero;
    if (lane == 31) sbuf[warp].x = ix;
    if (lane == 0) sbuf[warp].y = iy;
    __syncthreads();
    if (warp == 0) {
        T wx = lane < nw ? sbuf[lane].x : zero;
        T wy = lane < nw ? sbuf[lane].y : zero;
        T sx = warp_incl_scan<false>(wx, OpAdd());
        T sy = warp_incl_scan<true>(wy, OpAdd());
        T qx = shfl_up_t(sx, 1), qy = shfl_dn_t(sy, 1);
        if (lane == 0) qx = zero;
        if (lane == 31) qy = zero;
        __syncwarp();
        if (lane < nw) {
            sbuf[lane].x = qx;
            sbuf[lane].y = qy;
        }
        if (lane == 31) sbuf[32].x = sx;
        if (lane == 0) sbuf[32].y = sy;
    }
    __syncthreads();
    Pair<T> res = {acc_add(sbuf[warp].x, ex), acc_add(sbuf[warp].y, ey)};
    tx = sbuf[32].x;
    ty = sbuf[32].y;
    __syncthreads();
    return res;
}

// One-barrier forms of the two block scans above, with the same
// arithmetic in the same order (bitwise the same results): every warp scans
// the warp totals itself instead of warp 0 scanning them between two more
// barriers.  sbuf needs nw (not 33) values; every warp reads it after the
// one barrier, so it must not be written again before a later barrier:
// consecutive calls without a barrier between them alternate two buffers.
template <bool REV, class T, class Op>
__device__ __forceinline__ T block_excl_scan1(T v, Op op, T ident, T* sbuf, T& total) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T inc = warp_incl_scan<REV>(v, op);
    T lex = REV ? shfl_dn_t(inc, 1) : shfl_up_t(inc, 1);
    if (REV ? (lane == 31) : (lane == 0)) lex = ident;
    if (REV ? (lane == 0) : (lane == 31)) sbuf[warp] = inc;
    __syncthreads();
    T wv = lane < nw ? sbuf[lane] : ident;
    T winc = warp_incl_scan_n<REV>(wv, op, nw);
    T wex = REV ? shfl_dn_t(winc, 1) : shfl_up_t(winc, 1);
    if (REV ? (lane == 31) : (lane == 0)) wex = ident;
    total = shfl_idx_t(winc, REV ? 0 : scan_last_lane(nw));
    return op(shfl_idx_t(wex, warp), lex);
}

template <class T>
__device__ __forceinline__ Pair<T> block_excl_scan_fwd_rev1(T fx, T ry, T zero, Pair<T>* sbuf, T& tx, T& ty) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T ix = warp_incl_scan<false>(fx, OpAdd());
    T iy = warp_incl_scan<true>(ry, OpAdd());
    T ex = shfl_up_t(ix, 1), ey = shfl_dn_t(iy, 1);
    if (lane == 0) ex = zero;
    if (lane == 31) ey = zero;
    if (lane == 31) sbuf[warp].x = ix;
    if (lane == 0) sbuf[warp].y = iy;
    __syncthreads();
    T wx = lane < nw ? sbuf[lane].x : zero;
    T wy = lane < nw ? sbuf[lane].y : zero;
    T sx = warp_incl_scan_n<false>(wx, OpAdd(), nw);
    T sy = warp_incl_scan_n<true>(wy, OpAdd(), nw);
    T qx = shfl_up_t(sx, 1), qy = shfl_dn_t(sy, 1);
    if (lane == 0) qx = zero;
    if (lane == 31) qy = zero;
    tx = shfl_idx_t(sx, scan_last_lane(nw));
    ty = shfl_idx_t(sy, 0);
    return {acc_add(shfl_idx_t(qx, warp), ex), acc_add(shfl_idx_t(qy, warp), ey)};
}

// The exclusive sum of t and the exclusive forward and reverse products of
// mf and mr with one barrier (each as its own one-barrier scan would give
// it); totals in tt, and with TOT the products' in tf and tr.  The d_zeta psi
// sum and the B^(p) solve's matrices both depend on psi only.
template <class A, class R>
struct SumMats {
    A t;
    Mat2<R> f, r;
};
template <bool TOT, class Op = OpMatLeft, class A, class R>
__device__ __forceinline__ A block_excl_scan_sum_mats1(A t, Mat2<R> mf, Mat2<R> mr, A zero, SumMats<A, R>* sbuf,
                                                       Mat2<R>& ef, Mat2<R>& er, A& tt, Mat2<R>& tf, Mat2<R>& tr) {
    const Mat2<R> I2 = Op::template one<R>();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    A it = warp_incl_scan<false>(t, OpAdd());
    Mat2<R> ix = warp_incl_scan<false>(mf, Op());
    Mat2<R> iy = warp_incl_scan<true>(mr, Op());
    A et = shfl_up_t(it, 1);
    Mat2<R> ex = shfl_up_t(ix, 1), ey = shfl_dn_t(iy, 1);
    if (lane == 0) {
        et = zero;
        ex = I2;
        sbuf[warp].r = iy;
    }
    if (lane == 31) {
        ey = I2;
        sbuf[warp].t = it;
        sbuf[warp].f = ix;
    }
    __syncthreads();
    A wt = zero;
    Mat2<R> wx = I2, wy = I2;
    if (lane < nw) {
        wt = sbuf[lane].t;
        wx = sbuf[lane].f;
        wy = sbuf[lane].r;
    }
    A st = warp_incl_scan_n<false>(wt, OpAdd(), nw);
    Mat2<R> sx = warp_incl_scan_n<false>(wx, Op(), nw);
    Mat2<R> sy = warp_incl_scan_n<true>(wy, Op(), nw);
    const int last = scan_last_lane(nw);
    tt = shfl_idx_t(st, last);
    A qt = shfl_up_t(st, 1);
    Mat2<R> qx = shfl_up_t(sx, 1), qy = shfl_dn_t(sy, 1);
    if (lane == 0) {
        qt = zero;
        qx = I2;
    }
    if (lane == 31) qy = I2;
    ef = Op()(shfl_idx_t(qx, warp), ex);
    er = Op()(shfl_idx_t(qy, warp), ey);
    if (TOT) {
        tf = shfl_idx_t(sx, last);
        tr = shfl_idx_t(sy, 0);
    }
    return acc_add(shfl_idx_t(qt, warp), et);
}

// first index i in [0, n) with a[i] >= x (n if none)
template <class R>
__device__ __forceinline__ int lower_bound_dev(const R* a, int n, R x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

}  // namespace gbwake
