// ring_jump_host <rings> <rings per thread>: products of the ring matrices of
// csrc/ring_jump.cuh in the association of the register marches (a thread's
// rings one after the other, log-step scans over 32 lanes, over a block's 8
// warps and the blocks before), in float, against double of the same float
// matrices.  Prints, for the regular solution at the threads' first regions
// and the decaying one at their last, by how much its change over a distance
// of up to 1 is off (relative).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "ring_jump.cuh"

using namespace gbwake;
using M = Mat2<float>;

static double worst(const std::vector<double>& e, const std::vector<double>& at) {  // of e_t - e_s, |at_t - at_s| <= 1
    double w = 0;
    for (size_t t = 0; t < e.size(); ++t)
        for (size_t s = t + 1; s < e.size() && at[s] - at[t] <= 1.0; ++s) w = std::fmax(w, std::fabs(e[t] - e[s]));
    return w;
}

// exclusive products over threads 0, 1, ... of leaf[], as the marches scan them
static std::vector<M> scan(const std::vector<M>& leaf) {
    const OpMatDevLeft op;
    const M one = OpMatDevLeft::one<float>();
    const int W = 32, NW = 8;
    std::vector<M> out(leaf.size(), one);
    M before = one;  // of the blocks
    for (size_t b = 0; b < leaf.size(); b += W * NW) {
        std::vector<M> v(W * NW, one), tot(NW, one);
        for (size_t i = 0; i < v.size() && b + i < leaf.size(); ++i) v[i] = leaf[b + i];
        auto incl = [&](M* a, int n) {
            for (int o = 1; o < n; o <<= 1) {
                const std::vector<M> old(a, a + n);
                for (int i = o; i < n; ++i) a[i] = op(old[i - o], old[i]);
            }
        };
        for (int w = 0; w < NW; ++w) {
            incl(&v[w * W], W);
            tot[w] = v[w * W + W - 1];
        }
        incl(tot.data(), NW);
        for (int w = 0; w < NW; ++w)
            for (int l = 0; l < W && b + w * W + l < leaf.size(); ++l)
                out[b + w * W + l] = op(before, op(w ? tot[w - 1] : one, l ? v[w * W + l - 1] : one));
        before = op(before, tot[NW - 1]);
    }
    return out;
}

int main(int argc, char** argv) {
    const int n = atoi(argv[1]), K = atoi(argv[2]), T = (n + K - 1) / K;
    const double edge = 6.0;
    std::vector<float> r(n), A(n), m(n);
    for (int i = 0; i < n; ++i) {
        r[i] = (float)((i + 0.5) * edge / n);
        A[i] = (float)(edge / n * (i + 0.5) * edge / n) / r[i];  // w / r, psibar = 1
        m[i] = 0.5f * A[i] / r[i];
    }
    std::vector<M> f(T, OpMatDevLeft::one<float>()), b = f;
    for (int t = 0; t < T; ++t) {
        for (int i = t * K; i < n && i < (t + 1) * K; ++i) RingJump<float>(r[i], A[i], m[i]).multiply<false>(f[t]);
        for (int i = std::min(n, (t + 1) * K) - 1; i >= t * K; --i)
            RingJump<float>(r[i], A[i], m[i]).multiply<true>(b[T - 1 - t]);
    }
    const std::vector<M> F = scan(f), B = scan(b);
    // double: R from the axis outwards, D from beyond the last ring inwards
    std::vector<double> at(T), er(T), ed(T);
    double x0 = 1, x1 = 0;
    for (int t = 0; t < T; ++t) {
        at[t] = r[t * K];
        const double h0 = 1.0 + F[t].m00;
        er[t] = h0 / x0 - 1;
        for (int i = t * K; i < n && i < (t + 1) * K; ++i) RingJump<double>(r[i], A[i], m[i]).cross(x0, x1);
    }
    x0 = 0, x1 = 1;
    for (int t = T - 1; t >= 0; --t) {
        ed[t] = (1.0 + B[T - 1 - t].m11) / x1 - 1;
        for (int i = std::min(n, (t + 1) * K) - 1; i >= t * K; --i) RingJump<double>(r[i], A[i], m[i]).cross_back(x0, x1);
    }
    printf("%.3e %.3e\n", worst(er, at), worst(ed, at));
    return 0;
}
