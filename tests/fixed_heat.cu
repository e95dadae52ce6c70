// Host program of test_fixed_heat.py: blocks of values advanced one step by the
// integer arithmetic of exact64.cuh and by the FP64 operations.
//   fixed_heat <r> <kind> <blocks> <seed>
// prints: blocks the unit takes, blocks that failed, results that differ.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>

#include "exact64.cuh"

static double draw(std::mt19937_64 &g, const std::string &kind) {
    std::uniform_real_distribution<double> u(0.0, 1.0);
    const double x = u(g);
    if (kind == "one_binade") return 1.0 + x;
    if (kind == "negative") return -1.0 - x;
    if (kind == "two_binades") return 1.0 + 2.999 * x;
    if (kind == "binades") return std::exp2(6.0 * x - 3.0);              // six binades
    if (kind == "smooth") return 4.0 + 1e-3 * x;
    if (kind == "ties") return 1.0 + std::floor(x * 1048576.0) * 0x1p-52;
    if (kind == "few_bits") return 1.0 + std::floor(8.0 * x) / 8.0;
    if (kind == "powers") return std::exp2(std::floor(6.0 * x) - 3.0);
    if (kind == "smallest") return (1.0 + x) * 0x1p-1022;
    if (kind == "huge") return (1.0 + x) * 0x1p1015;
    exit(2);
}

static int upper(double v) {
    long long b;
    memcpy(&b, &v, 8);
    return (int)(b >> 32);
}

int main(int, char **argv) {
    const double r = atof(argv[1]);
    const std::string kind = argv[2];
    std::mt19937_64 g(atoi(argv[4]));
    long long taken = 0, failed = 0, differ = 0;
    const int n = 12;
    double u[n][n];
    for (int b = 0; b < atoi(argv[3]); ++b) {
        int high = INT_MIN, low = INT_MAX;
        for (auto &row : u)
            for (double &v : row) {
                v = draw(g, kind);
                high = upper(v) > high ? upper(v) : high;
                low = upper(v) < low ? upper(v) : low;
            }
        swept::FixedHeat f;
        if (!f.fits(swept::heat_ratio(r), high, low)) continue;
        ++taken;
        long long bad = 0;
        for (int y = 1; y + 1 < n; ++y)
            for (int x = 1; x + 1 < n; ++x) {
                const double c = u[y][x], pe = u[y][x + 1] + u[y + 1][x], pw = u[y][x - 1] + u[y - 1][x];
                const double want = std::fma(r, std::fma(-4.0, c, pe + pw), c);
                const long long v =
                    f.next(f.from(c), f.sum(f.from(u[y][x + 1]), f.from(u[y + 1][x])),
                           f.sum(f.from(u[y][x - 1]), f.from(u[y - 1][x])));
                const double got = f.to(v);
                bad += memcmp(&got, &want, 8) != 0;
            }
        if (f.failed())
            ++failed;
        else
            differ += bad;
    }
    printf("%lld %lld %lld\n", taken, failed, differ);
    return 0;
}
