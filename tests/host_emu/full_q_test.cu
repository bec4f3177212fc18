// CPU test of the float32 shortcut to the full covariance's q (full_q_f32):
// wherever it claims a granularity beyond doubt, that must be the granularity
// of the quotient in 64 bits, with the division two units in the last place
// off either way.  Sweeps visibility scales over everything that is accepted,
// with q placed near powers of four, nearly cancelling sums among them.
#include <cstdio>
#include <random>
#include <vector_types.h>
#include "../../paper_1503_00638_gb300/csrc/common.cuh"
using namespace bsg;

int main()
{
    std::mt19937_64 g(5);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    uint64_t accepted = 0, ordinary = 0, ordinary_accepted = 0;
    for (int scale10 = -20; scale10 <= 22; scale10++)
        for (double N : {1.0, 65536.0, 1e9, 1.2e10, 1e25})
            for (int it = 0; it < 20000; it++) {
                // W = C^-1-like: 1 / |V| of both inputs, a correlation below one
                const double s = pow(10.0, -scale10), wi = s * (0.5 + U(g)), wj = s * pow(10.0, 4.0 * U(g) - 2.0);
                const double rho = it & 1 ? U(g) : 1.0 - pow(10.0, -6.0 * U(g)), ph = 6.283185307179586 * U(g);
                const double wr = rho * sqrt(wi * wj) * cos(ph), wm = rho * sqrt(wi * wj) * sin(ph);
                const bool is_auto = it % 5 == 0;
                const int part = is_auto ? 0 : it & 1;
                const double re2 = wr * wr - wm * wm, ww = is_auto ? wi * wi : wi * wj;
                const double h = is_auto ? N * ww : 2.0 * N * (part ? ww - re2 : ww + re2);
                // f such that q lies a little beside 4^k
                const int k = (int)(g() % 96) - 48;
                const double d = pow(10.0, -1.0 - 6.5 * U(g)) * (g() & 1 ? 1 : -1);
                const double f = pow(4.0, k) * (1.0 + d) * h / 12.0;
                if (!(h > 0) || !(f >= 0) || !std::isfinite(f) || !std::isfinite(1.0 / h)) continue;
                const float q64 = (float)(12.0 * f * (1.0 / h));
                const float f12 = (float)(12.0 * f / N);
                float q;
                const bool sure = full_q_f32(f12, (float)wi, (float)(is_auto ? wi : wj), is_auto ? 0.f : (float)wr,
                                             is_auto ? 0.f : (float)wm, is_auto, part, q);
                // whole magnitudes: visibilities of 1e-3 to 1e4, f / N of 1e-9 and more, d of 1e-3 and more
                if (scale10 >= -3 && scale10 <= 4 && f / N > 1e-9 && f / N < 1 && fabs(d) > 1e-3 && rho < 0.9) {
                    ordinary++;
                    ordinary_accepted += sure;
                }
                if (!sure) continue;
                accepted++;
                for (int off = -2; off <= 2; off++)
                    if (!q_usable(float_bits(q64)) || magic_bits(float_bits(q) + off) != magic_bits(float_bits(q64))) {
                        printf("scale 1e%d, N %g, f %g: q %.9g for %.9g (h %.3g, f12 %.3g)\n", scale10, N, f, q, q64,
                               h / N, f12);
                        return 1;
                    }
            }
    printf("%llu accepted, of ordinary ones %llu of %llu\n", (unsigned long long)accepted,
           (unsigned long long)ordinary_accepted, (unsigned long long)ordinary);
    return accepted < 100000 || ordinary_accepted < ordinary * 9 / 10;
}
