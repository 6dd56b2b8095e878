// Host check of the moment bounds with 6 / 8 power and 3 / 4 trigonometric
// moments: absorbers along rays (a few Gaussian bumps of absorbance over part
// of the depth range, with or without a floor), their float32 moments, and the
// fraction A in front at sampled depths in the library's float32 arithmetic,
// compiled with the host compiler.  One line per depth: z, the four A, the
// nine power moments, the four complex trigonometric moments.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "mboit_power.cuh"

using namespace mb;

// As the library fills them: coefficients of s^m in (s + i)^k (s - i)^(n - k).
static void fill(TrigTables& T, int n) {
    std::memset(&T, 0, sizeof T);
    T.n = n;
    T.zone_scale = (float)(0.9 * 3.14159265358979323846);
    for (int k = 0; k <= n; ++k) {
        double cr[6] = {1}, ci[6] = {0};
        for (int f = 0; f < n; ++f) {
            const double rim = f < k ? 1 : -1;
            double nr[6] = {0}, ni[6] = {0};
            for (int m = 0; m <= f; ++m) {
                nr[m + 1] += cr[m];
                ni[m + 1] += ci[m];
                nr[m] -= ci[m] * rim;
                ni[m] += cr[m] * rim;
            }
            std::memcpy(cr, nr, sizeof cr);
            std::memcpy(ci, ni, sizeof ci);
        }
        for (int m = 0; m <= n; ++m) {
            T.er[k][m] = (float)cr[m];
            T.ei[k][m] = (float)ci[m];
        }
    }
}

int main() {
    std::mt19937_64 rng(5);
    std::uniform_real_distribution<double> U(0, 1);
    TrigTables T3, T4;
    fill(T3, 3);
    fill(T4, 4);
    for (int it = 0; it < 300; ++it) {
        const int n = 20 + (int)(U(rng) * 400), nb = 1 + (int)(U(rng) * 5);
        const double za = U(rng) * 1.6 - 0.9, zb = za + (0.05 + U(rng)) * (0.95 - za);
        double c[5], s[5], h[5], m[9] = {0}, tr[4] = {0}, ti[4] = {0};
        for (int j = 0; j < nb; ++j) {
            c[j] = za + (zb - za) * U(rng);
            s[j] = (zb - za) * (0.02 + 0.3 * U(rng));
            h[j] = U(rng);
        }
        const double base = U(rng) < 0.5 ? 0 : 0.05 * U(rng);
        std::vector<double> zs;
        for (int i = 0; i < n; ++i) {
            const double z = (float)(za + (zb - za) * (i + .5) / n);
            double a = base;
            for (int j = 0; j < nb; ++j) a += h[j] * std::exp(-(z - c[j]) * (z - c[j]) / (2 * s[j] * s[j]));
            a *= 0.05;
            double p = a;
            for (int j = 0; j < 9; ++j, p *= z) m[j] += p;
            for (int j = 0; j < 4; ++j) {
                tr[j] += a * std::cos((j + 1) * 0.9 * M_PI * z);
                ti[j] += a * std::sin((j + 1) * 0.9 * M_PI * z);
            }
            zs.push_back(z);
        }
        float fm[9];
        cf tau[4];
        for (int j = 0; j < 9; ++j) fm[j] = (float)m[j];
        for (int j = 0; j < 4; ++j) tau[j] = {(float)(tr[j] / m[0]), (float)(ti[j] / m[0])};
        const auto P3 = make_power_frame<3>(fm, 5e-5f);
        const auto P4 = make_power_frame<4>(fm, 5e-5f);
        const TrigFrame F3 = make_trig_frame(fm[0], tau, 3, 2e-3f), F4 = make_trig_frame(fm[0], tau, 4, 2e-3f);
        for (int q = 0; q < 8; ++q) {
            const float z = (float)zs[(int)(U(rng) * n)];
            std::printf("%.9g %.9g %.9g %.9g %.9g", z, power_fraction<3>(P3, z, .3f), power_fraction<4>(P4, z, .3f),
                        trig_fraction<3, float>(F3, T3, z, .3f), trig_fraction<4, float>(F4, T4, z, .3f));
            for (int j = 0; j < 9; ++j) std::printf(" %.9g", fm[j]);
            for (int j = 0; j < 4; ++j) std::printf(" %.9g %.9g", tau[j].x, tau[j].y);
            std::printf("\n");
        }
    }
}
