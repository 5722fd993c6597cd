// The on-chip re-sort's steps (csrc/key_sort.cuh) run over T emulated threads in the order resort() takes them:
// registers, neighbour rounds, pairwise merges.  argv: rings per thread, kind of radii.  Every access is checked;
// the result is compared with std::sort of the (bit pattern, position) pairs.
#include "key_sort.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <random>
#include <string>
#include <vector>

using namespace gbwake;

static int32_t key_of(float r) {
    r += 0.f;
    int32_t k;
    std::memcpy(&k, &r, 4);
    return k;
}

static std::vector<float> radii(int n, const std::string& kind, unsigned seed) {
    std::mt19937 rng(seed);
    std::vector<float> r(n);
    for (int i = 0; i < n; ++i) r[i] = (i + 0.5f) / n;
    const float nan = std::numeric_limits<float>::quiet_NaN(), inf = std::numeric_limits<float>::infinity();
    if (kind == "near")
        for (int i = 0; i + 1 < n; i += 3) std::swap(r[i], r[i + 1]);
    if (kind == "reversed") std::reverse(r.begin(), r.end());
    if (kind != "near" && kind != "reversed") std::shuffle(r.begin(), r.end(), rng);
    if (kind == "ties")
        for (float& x : r) x = std::floor(8.f * x) / 8.f;
    if (kind == "one nan") {  // a ring without a number, one that crossed from end to end, the others in order
        std::sort(r.begin(), r.end());
        std::swap(r[0], r[n - 1]);
        r[rng() % n] = nan;
    }
    if (kind == "nan and inf")
        for (float& x : r) x = rng() % 4 == 0 ? nan : rng() % 8 == 0 ? inf : rng() % 16 == 0 ? -nan : rng() % 16 == 0 ? -0.f : x;
    if (kind == "all nan") std::fill(r.begin(), r.end(), nan);
    return r;
}

template <int K>
static bool run(int T, int n, const std::string& kind, int near_rounds, unsigned seed) {
    const int TK = T * K;
    const std::vector<float> r = radii(n, kind, seed);
    std::vector<KeySrc> tab(TK), other(TK);
    std::vector<KeySrc> want(TK);
    for (int p = 0; p < TK; ++p) want[p] = {p < n ? key_of(r[p]) : kNoRingKey, p};
    auto less = [](const KeySrc& a, const KeySrc& b) { return a.key != b.key ? a.key < b.key : a.src < b.src; };
    std::vector<KeySrc> v = want;
    std::sort(want.begin(), want.end(), less);
    auto regs = [&](int t, auto f) {
        KeySrc x[K];
        for (int k = 0; k < K; ++k) x[k] = v.at(t * K + k);
        f(x);
        for (int k = 0; k < K; ++k) v.at(t * K + k) = x[k];
    };
    for (int t = 0; t < T; ++t) regs(t, [](KeySrc(&x)[K]) { ks_sort<K>(x); });
    bool sorted = false;
    for (int round = 0; round <= near_rounds && !sorted; ++round) {
        tab = v;
        sorted = true;
        for (int t = 0; t + 1 < T; ++t)
            if (ks_less(tab.at((t + 1) * K), v.at(t * K + K - 1))) sorted = false;
        if (sorted || round == near_rounds) break;
        for (int t = 0; t < T; ++t) {
            const bool left = (t & 1) == (round & 1);
            const int partner = left ? t + 1 : t - 1;
            if (partner >= 0 && partner < T)
                regs(t, [&](KeySrc(&x)[K]) {
                    ks_merge_split<K>(x, [&](int k) { return tab.at(partner * K + k); }, left);
                });
        }
    }
    if (!sorted)
        for (int L = K; L < TK; L <<= 1) {
            for (int t = 0; t < T; ++t) {
                const int p0 = t * K, base = p0 & ~(2 * L - 1);
                const int nA = std::min(L, TK - base), nB = std::max(0, std::min(L, TK - base - L));
                ks_merge_outputs<K>(
                    [&](int i) {
                        if (!(i >= 0 && i < nA) && !(i >= L && i < L + nB)) std::printf("run index %d\n", i), std::exit(1);
                        return tab.at(base + i);
                    },
                    L, nA, nB, p0 - base, [&](int k, KeySrc e) { other.at(p0 + k) = e; });
            }
            std::swap(tab, other);
        }
    for (int p = 0; p < TK; ++p)
        if (tab[p].src != want[p].src || tab[p].key != want[p].key || (p < n && !(tab[p].src >= 0 && tab[p].src < n))) {
            std::printf("K %d T %d n %d %s rounds %d seed %u: place %d holds position %d, not %d\n", K, T, n, kind.c_str(),
                        near_rounds, seed, p, tab[p].src, want[p].src);
            return false;
        }
    return true;
}

int main(int, char** argv) {
    const int K = std::atoi(argv[1]);
    bool ok = true;
    for (int T : {32, 64, 96, 512})
        for (int n : {1, 2, 31, T * K / 2 + 1, T * K - 3, T * K})
            for (int rounds : {0, 8})
                for (unsigned seed = 0; seed < 6; ++seed)
                    ok = ok && (K == 2 ? run<2> : K == 4 ? run<4> : run<8>)(T, n, argv[2], rounds, seed);
    return ok ? 0 : 1;
}
