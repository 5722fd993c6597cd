// csrc/f64_log.cuh on the host against long double arithmetic (64 bits of significand or more): prints the largest
// errors in ulp over the range of doubles and around 1; exit 1 where a special value differs from the library's.
#include "f64_log.cuh"

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>

using namespace gbwake;
static constexpr F64LogTable kTable = f64_log_table();

static double err(double x) {
    const long double want = logl((long double)x);
    int e;
    frexp((double)want, &e);
    return (double)(fabsl((long double)f64_log(kTable, x) - want) / ldexpl(1.0L, e - 53));
}

int main() {
    std::mt19937_64 rng(7);
    double all = 0.0, radii = 0.0, near = 0.0, edges = 0.0;
    auto up = [](double& m, double v) {
        if (!(v <= m)) m = v;
    };
    for (int k = 0; k < 3000000; ++k) {
        const uint64_t b = rng() & 0x7fffffffffffffffull;
        double x;
        std::memcpy(&x, &b, 8);
        if (std::isnormal(x)) up(all, err(x));
        up(radii, err(1e-6 * std::pow(1e9, (double)(rng() >> 11) * 0x1p-53)));
        x = 1.0 + std::ldexp((double)(int64_t)rng(), -63 - (int)(rng() % 52));
        if (x > 0.0 && x != 1.0) up(near, err(x));
    }
    for (int i = 0; i < 128; ++i)  // the table's intervals end to end, for several exponents
        for (int ex : {-1022, -40, -2, -1, 0, 1, 2, 40, 1023})
            for (uint64_t low : {0ull, 1ull, 0x0fffffffffffull, 0x1fffffffffffull}) {
                const uint64_t b = (uint64_t)(ex + 1023) << 52 | (uint64_t)i << 45 | low;
                double x;
                std::memcpy(&x, &b, 8);
                if (x != 1.0) up(edges, err(x));
            }
    std::printf("%.6f %.6f %.6f %.6f\n", all, radii, near, edges);
    const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
    bool ok = f64_log(kTable, 1.0) == 0.0 && f64_log(kTable, inf) == inf && f64_log(kTable, 0.0) == -inf;
    ok = ok && std::isnan(f64_log(kTable, -1.0)) && std::isnan(f64_log(kTable, nan)) && std::isnan(f64_log(kTable, -inf));
    ok = ok && f64_log(kTable, 5e-324) == std::log(5e-324);
    return ok ? 0 : 1;
}
