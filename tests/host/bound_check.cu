// Host check of cmp_bound_terms as the library computes it: for tables of 27 and of 9 cells at class
// sizes from balanced to empty and up to 131072 samples -- spread evenly, concentrated, associated, and
// with the cells where the bound is tightest -- the bound of the float constants, in FP32 like the
// kernels', never exceeds K2 (log-gamma, long double), and is not looser than its slack and the
// parabola's give-away explain (a constant that drifts shows either way).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "../../paper_2201_10956_gb300/csrc/epi3_internal.cuh"

using namespace epi3;

static unsigned long long state = 88172645463325252ull;
static double uni() {
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return (double)(state >> 11) / 9007199254740992.0;
}

int main() {
    const int sizes[][2] = {{1, 0}, {0, 1}, {50, 50}, {700, 300}, {30, 970}, {4096, 4096}, {9000, 3000},
                            {131072, 0}, {131071, 1}, {131000, 72}, {65536, 65536}, {100000, 31072}, {5, 131067}};
    long long tables = 0;
    double closest = 1e300;
    for (const auto& nc : sizes) {
        const int N = nc[0] + nc[1];
        int e2 = 0;
        std::frexp(std::lgamma((double)N + 2.0), &e2);
        const CmpBoundTerms B = cmp_bound_terms(nc[0], nc[1], std::ldexp(1.0f, -23), std::ldexp(1.0f, e2 - 36));
        for (int cells : {27, 9})
            for (int rep = 0; rep < 4000; ++rep) {
                // cell weights, then the samples of each class dealt by them
                std::vector<double> w(cells), a(cells);
                double sw[2] = {0.0, 0.0};
                const int shape = rep % 4;
                for (int q = 0; q < cells; ++q) {
                    w[q] = shape == 0 ? 1.0 : shape == 1 ? std::pow(uni(), 6.0) : shape == 2 ? (uni() < 0.2) : uni();
                    a[q] = shape == 3 ? std::exp(3.0 * (uni() - 0.5)) : 1.0;   // association
                    sw[0] += w[q];
                    sw[1] += w[q] * a[q];
                }
                std::vector<int> r[2] = {std::vector<int>(cells, 0), std::vector<int>(cells, 0)};
                for (int c = 0; c < 2; ++c) {
                    int left = nc[c];
                    for (int q = 0; q < cells && sw[c] > 0; ++q) {
                        const double f = w[q] * (c ? a[q] : 1.0) / sw[c];
                        const int n = std::min(left, (int)std::lround(f * nc[c] + (rep % 3 ? 2.0 * uni() - 1.0 : 0.0)));
                        r[c][q] = std::max(n, 0);
                        left -= r[c][q];
                    }
                    r[c][(int)(uni() * cells)] += left;
                }
                long double k2 = 0.0L;
                float sum = 0.f, lgs = 0.f;
                for (int q = 0; q < cells; ++q) {
                    k2 += lgammal(r[0][q] + r[1][q] + 2.0L) - lgammal(r[0][q] + 1.0L) - lgammal(r[1][q] + 1.0L);
                    const float us = (float)(r[0][q] + r[1][q] + 2), um = (float)(r[B.minor][q] + 1);
                    const float quo = um * um / us;
                    if (cells == 27) {
                        sum += quo;
                        lgs += std::log2(us);
                    } else {
                        sum += um - quo;
                        lgs += std::log2(um - quo);
                    }
                }
                const float b = cells == 27 ? std::fmaf(-B.c, sum, 0.34657359f * lgs) : std::fmaf(B.c, sum, 0.34657359f * lgs);
                const double bound = (double)b - (double)(cells == 27 ? B.off : B.off2);
                ++tables;
                closest = std::min(closest, (double)k2 - bound);
                if (bound > (double)k2) {
                    std::printf("bound %.6f above K2 %.6f: classes %d %d, %d cells, table %d\n", bound, (double)k2,
                                nc[0], nc[1], cells, rep);
                    return 1;
                }
                if (shape == 0 && N >= 100 && (double)k2 - bound > 60.0 + 2.0 * B.slack) {
                    std::printf("bound %.6f far below K2 %.6f: classes %d %d, %d cells, table %d\n", bound, (double)k2,
                                nc[0], nc[1], cells, rep);
                    return 1;
                }
            }
    }
    std::printf("bound ok: %lld tables, closest %.4f nats\n", tables, closest);
    return 0;
}
