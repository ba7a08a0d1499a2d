// CPU check of the FP32-word sums (csrc/esp_dd.h) against the FP64 tile code
// and an extended-precision sum of the same records.  Arguments: seed.  Prints
// one line per form: name, records, largest |words - exact| and |FP64 - exact|
// over the sum of absolute terms.
#include <vector_types.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "esp_dd.h"
#include "esp_eval_core.h"

using namespace esp;
using real = long double;

// sum_h G_h S_h of a record where its Gaussian is negligible (asymptotic Boys
// values), by the Hermite recursion
static real far_exact(int L, const double *r, const double *c, real &mag)
{
    const real sp = r[3], x = sp * (real(r[0]) - c[0]), y = sp * (real(r[1]) - c[1]), z = sp * (real(r[2]) - c[2]);
    const real T = x * x + y * y + z * z;
    real S[kMaxL + 1][35];
    for (int n = L; n >= 0; --n) {
        real f = 0.886226925452758013649083741670572591L / sqrtl(T);
        for (int k = 0; k < n; ++k)
            f *= -(2 * k + 1) / T; // (-2)^n F_n
        S[n][0] = f;
        for (int N = 1; N <= L - n; ++N)
            for (int t = N; t >= 0; --t)
                for (int u = N - t; u >= 0; --u) {
                    const int v = N - t - u;
                    real w;
                    if (t > 0)
                        w = x * S[n + 1][hidx(t - 1, u, v)] + (t > 1 ? (t - 1) * S[n + 1][hidx(t - 2, u, v)] : 0);
                    else if (u > 0)
                        w = y * S[n + 1][hidx(t, u - 1, v)] + (u > 1 ? (u - 1) * S[n + 1][hidx(t, u - 2, v)] : 0);
                    else
                        w = z * S[n + 1][hidx(t, u, v - 1)] + (v > 1 ? (v - 1) * S[n + 1][hidx(t, u, v - 2)] : 0);
                    S[n][hidx(t, u, v)] = w;
                }
    }
    real s = 0;
    for (int h = 0; h < num_hermite(L); ++h) {
        s += r[4 + h] * S[0][h];
        mag += fabsl(r[4 + h] * S[0][h]);
    }
    return s;
}

template <int L>
static double far_words(const DdTile &t, const DdPos &c)
{
    TdSum s;
    s.clear();
    f2 r2;
    for (int j = 0; j < t.n4; j += 2)
        td_far<L>(t, j, c, true, true, s, r2);
    return s.total();
}

static double words_sum(int cls, const DdTile &t, const DdPos &c)
{
    if (is_point_class(cls)) {
        TdSum s;
        s.clear();
        f2 r2;
        for (int j = 0; j < t.n4; j += 2)
            td_point(t, j, c, s, r2);
        return s.total();
    }
    switch (cls & 7) {
    case 0: return far_words<0>(t, c);
    case 1: return far_words<1>(t, c);
    case 2: return far_words<2>(t, c);
    case 3: return far_words<3>(t, c);
    default: return far_words<4>(t, c);
    }
}

int main(int argc, char **argv)
{
    std::mt19937_64 gen(argc > 1 ? atoi(argv[1]) : 1);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    const double q = 0x1p-17, spread = 30.0; // 2^24 q > 4 max |P|
    const int classes[] = {kClassPoint, 0, 1, 2, 3, 4};
    const int sizes[] = {1, 2, 3, 5, 8};
    for (int cls : classes)
        for (int n : sizes) {
            const int L = is_point_class(cls) ? 0 : cls, st = is_point_class(cls) ? kPointStride64 : rec64_stride(L);
            double worst = 0.0, worst64 = 0.0;
            for (int rep = 0; rep < 200; ++rep) {
                TileMeta m;
                std::memset(&m, 0, sizeof m);
                m.cls = cls;
                m.n = n;
                std::vector<double> rec(size_t(n) * st, 0.0);
                for (int j = 0; j < n; ++j) {
                    double *r = &rec[size_t(j) * st];
                    for (int k = 0; k < 3; ++k)
                        r[k] = rep % 4 == 0 ? std::ldexp(std::round(u(gen) * 64), -1) : rep % 4 == 1 ? u(gen) * 1e-9 : spread * u(gen);
                    r[3] = is_point_class(cls) ? std::pow(10.0, 3 * u(gen)) * (u(gen) < 0 ? -1 : 1) : 8.0 + 4.0 * u(gen);
                    for (int h = 0; h < (is_point_class(cls) ? 0 : num_hermite(L)); ++h)
                        r[4 + h] = u(gen);
                }
                double c[3];
                real d2 = 0;
                do { // every record far: T >= 16 x 6^2
                    for (int k = 0; k < 3; ++k)
                        c[k] = spread * u(gen);
                    d2 = 1e300;
                    for (int j = 0; j < n; ++j) {
                        real s = 0;
                        for (int k = 0; k < 3; ++k)
                            s += (real(rec[size_t(j) * st + k]) - c[k]) * (real(rec[size_t(j) * st + k]) - c[k]);
                        d2 = std::min(d2, s);
                    }
                } while (d2 < 36);
                const int n4 = dd_pad(n);
                std::vector<float> w(size_t(n4) * dd_words(m), 0.0f);
                for (int j = 0; j < n4; ++j) {
                    dd_convert(m, &rec[size_t(std::min(j, n - 1)) * st], q, w.data() + j, n4);
                    if (j >= n)
                        dd_zero_coefficients(m, w.data() + j, n4);
                }
                DdPos p;
                for (int k = 0; k < 3; ++k)
                    dd_split3(c[k], q, 1 / q, p.h[k], p.m[k], p.l[k]);
                real exact = 0, mag = 0;
                for (int j = 0; j < n; ++j) {
                    const double *r = &rec[size_t(j) * st];
                    if (is_point_class(cls)) {
                        real s = 0;
                        for (int k = 0; k < 3; ++k)
                            s += (real(r[k]) - c[k]) * (real(r[k]) - c[k]);
                        exact += r[3] / sqrtl(s);
                        mag += fabsl(r[3] / sqrtl(s));
                    } else {
                        exact += far_exact(L, r, c, mag);
                    }
                }
                double f64;
                if (is_point_class(cls)) {
                    const double c1[1][3] = {{c[0], c[1], c[2]}};
                    double a[1] = {0.0};
                    tile_points_f64<1>(rec.data(), n, c1, a);
                    f64 = a[0];
                } else {
                    f64 = tile_f64_one_any(cls, rec.data(), n, c[0], c[1], c[2], nullptr);
                }
                const double words = words_sum(cls, DdTile{w.data(), n4}, p);
                worst = std::max(worst, double(fabsl(words - exact) / mag));
                worst64 = std::max(worst64, double(fabsl(f64 - exact) / mag));
            }
            std::printf("%d %d %.3e %.3e\n", cls, n, worst, worst64);
        }
    return 0;
}
