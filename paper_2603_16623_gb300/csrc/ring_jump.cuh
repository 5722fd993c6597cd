// ring_jump.cuh -- a ring's jump matrix of the B_theta^(p) system, and products
// of such matrices that keep what differs from the identity.
//
// The matrix is I + h (1, -r^2)^T (r, 1/r) with h = A / 2 (A: Eq. b_coeffs_1),
// its inverse the same with -h.  One ring's h r is ~1e-3: rounded as it is,
// 1 + h r takes an error of up to 2^-24 that over alike rings has one sign,
// and in which march it cancels is a matter of the products' association and
// of what the compiler fuses.  Here the matrices are multiplied less the
// identity and the solutions walked across a ring by what it adds to them, so
// that errors are relative to the difference.  The mixed march of beam-grid
// wakes (march_reg_kernel) takes its products so at 3 and 4 rings per thread
// (its automatic shapes above 512 rings): with the matrices as they are it had
// lost precision against the global-memory march above 4096 rings.  E_z
// against 64 bits there, over 20 solves, median 1.1e-6 -> 2.2e-7 and largest
// 1.9e-6 -> 6.7e-7 (the global-memory march 4.2e-7 and 1.3e-6), B_theta
// 2.5e-7 -> 1.4e-7 (2.8e-7).  12 operations for a product of two, where the
// matrices as they are take 8, and no exchange of R between threads: 24 wakes
// 9.86 -> 9.92 ms (10.08 with this form above 4096 rings only: two kernels'
// instructions to fetch instead of one's).
// The other marches keep the matrices as they are.  FP64 (AB2, ions, RK4): the
// errors are those of the global-memory marches, and 12 FP64 operations for 8
// take 6 % on their pipe.  Mixed ions and RK4: E_z's error is 0.97 to 1.0 of
// the global-memory marches' up to 2048 rings, 1.7 from there to 4096 and 0.9
// above (RK4); this form brings 0.6 over all, but in their scans rings cross,
// both are 4e-4 from 64 bits, and any other rounding moves single particles'
// fields by 1e-2 to 1e-1: the results stay what they are.
// Compiles for the host too (tests).
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define WK_JUMP_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define WK_JUMP_HD inline
using std::fma;
#endif

namespace gbwake {

template <class R>
struct Mat2 {
    R m00, m01, m10, m11;
};

// a, applied first, then b, all less the identity: (I + b)(I + a) - I
struct OpMatDevLeft {
    template <class R>
    WK_JUMP_HD Mat2<R> operator()(Mat2<R> a, Mat2<R> b) const {
        return {fma(b.m00, a.m00, fma(b.m01, a.m10, a.m00 + b.m00)), fma(b.m00, a.m01, fma(b.m01, a.m11, a.m01 + b.m01)),
                fma(b.m10, a.m00, fma(b.m11, a.m10, a.m10 + b.m10)), fma(b.m10, a.m01, fma(b.m11, a.m11, a.m11 + b.m11))};
    }
    static constexpr bool kDev = true;
    template <class R>
    WK_JUMP_HD static Mat2<R> one() { return {0, 0, 0, 0}; }
    template <class R>
    WK_JUMP_HD static Mat2<R> whole(Mat2<R> m) { return {(R)1 + m.m00, m.m01, m.m10, (R)1 + m.m11}; }
};

template <class R>
struct RingJump {
    R hr, hi, r2;  // h r, h / r, r^2
    WK_JUMP_HD RingJump(R r, R A, R h_over_r) : hr((R)0.5 * A * r), hi(h_over_r), r2(r * r) {}
    // the solution x from below the ring to above it, and back
    WK_JUMP_HD void cross(R& x0, R& x1) const {
        const R q = fma(hr, x0, hi * x1);
        x0 += q;
        x1 = fma(-r2, q, x1);
    }
    WK_JUMP_HD void cross_back(R& x0, R& x1) const {
        const R q = fma(hr, x0, hi * x1);
        x0 -= q;
        x1 = fma(r2, q, x1);
    }
    // the matrix (BACK: its inverse) times I + m, less I
    template <bool BACK>
    WK_JUMP_HD void multiply(Mat2<R>& m) const {
        const R q0 = fma(hr, m.m00, fma(hi, m.m10, hr)), q1 = fma(hr, m.m01, fma(hi, m.m11, hi));
        if (BACK) m = {m.m00 - q0, m.m01 - q1, fma(r2, q0, m.m10), fma(r2, q1, m.m11)};
        else m = {m.m00 + q0, m.m01 + q1, fma(-r2, q0, m.m10), fma(-r2, q1, m.m11)};
    }
};

}  // namespace gbwake
