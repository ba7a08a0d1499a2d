// CPU check of one order at a time: far-form records whose coefficients of all
// other orders are zero (products without a monopole, for instance).  Argument:
// seed.  Prints per (L, order): root mean square of (words - exact) and of
// (FP64 code - exact) over the sum of absolute terms.
#define main words_check_main
#include "words_check.cpp"
#undef main

template <int L>
static void orders(std::mt19937_64 &gen)
{
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    const double q = 0x1p-18;
    TileMeta m;
    std::memset(&m, 0, sizeof m);
    m.cls = L;
    m.n = 1;
    for (int N = 0; N <= L; ++N) {
        double s2 = 0.0, s2_64 = 0.0;
        const int reps = 4000;
        for (int rep = 0; rep < reps; ++rep) {
            double r[rec64_stride(L)] = {}, c[3], d2 = 0.0;
            for (int k = 0; k < 3; ++k)
                r[k] = 12.0 * u(gen);
            r[3] = std::exp(2.0 + 2.0 * u(gen));
            do { // T from 46 up
                d2 = 0.0;
                for (int k = 0; k < 3; ++k) {
                    c[k] = r[k] + 40.0 / r[3] * u(gen);
                    d2 += (r[k] - c[k]) * (r[k] - c[k]);
                }
            } while (r[3] * r[3] * d2 < 46.0);
            for (int h = N * (N + 1) * (N + 2) / 6; h < (N + 1) * (N + 2) * (N + 3) / 6; ++h)
                r[4 + h] = u(gen);
            std::vector<float> w(size_t(4) * dd_words(m), 0.0f);
            for (int j = 0; j < 4; ++j) {
                dd_convert(m, r, q, w.data() + j, 4);
                if (j > 0)
                    dd_zero_coefficients(m, w.data() + j, 4);
            }
            DdPos p;
            for (int k = 0; k < 3; ++k)
                dd_split3(c[k], q, 1 / q, p.h[k], p.m[k], p.l[k]);
            real mag = 0;
            const real exact = far_exact(L, r, c, mag);
            const real e = (words_sum(L, DdTile{w.data(), 4}, p) - exact) / mag;
            const real e64 = (tile_f64_one_any(L, r, 1, c[0], c[1], c[2], nullptr) - exact) / mag;
            s2 += double(e * e);
            s2_64 += double(e64 * e64);
        }
        std::printf("%d %d %.3e %.3e\n", L, N, std::sqrt(s2 / reps), std::sqrt(s2_64 / reps));
    }
}

int main(int argc, char **argv)
{
    std::mt19937_64 gen(argc > 1 ? atoi(argv[1]) : 1);
    orders<0>(gen);
    orders<1>(gen);
    orders<2>(gen);
    orders<3>(gen);
    orders<4>(gen);
    return 0;
}
