// The FP64 sums in pairs of FP32 numbers.
//
// GB300's FP64 pipe runs at 1/63 of the FP32 rate (measured: a DADD occupies a
// scheduler for 64 cycles or more, an FFMA2 of two lanes for 2), so a value
// carried as an unevaluated sum h + l of two FP32 numbers (about 48 bits), with
// the error-free transformations of Knuth (TwoSum) and Dekker / FMA
// (TwoProduct), is far cheaper than one FP64 number.  Two records of a tile
// share each packed FP32 instruction (the lanes of an f2), one position per
// thread.
//
// Inputs lose nothing: every coordinate is stored as three FP32 words
//   x = h + m + l,  h on the environment's coordinate grid q,  m on the grid
//   q 2^-23,  l the rest (below 2^-24 q, so the sum holds x to 2^-48 q),
// and offsets are formed word by word: h and m differences are exact (each
// needs at most 24 bits of its grid), so P - C is exact to 2^-47 q before it is
// rounded once to 48 bits.  The terms of a few records are summed as pairs and
// go to FP64 accumulators.
//
// Far form (every Gaussian of the tile negligible at the position): a Hermite
// distribution's potential is sum_N F_N P_N(d) / r^(2N+1) with P_N the
// harmonic projection of its order-N moments (trace parts drop out because
// 1/r is harmonic), so a record stores per order the coefficients of
// (-1)^N (2N-1)!! P_N and the sum is a Horner scheme in 1/r^2.
// General form (L <= 2): the Hermite sum in scaled offsets x = sqrt(p) d with
// the Boys values from a Taylor table or their asymptotic form.
//
// A dd tile holds word w of record j at w * n4 + j, n4 = n rounded up to 4 (the
// padding repeats the last record's coordinates with zero coefficients):
//   0..2 h(x, y, z)   3..5 m   6..8 l
//   points:        9..11 Z (three words), 12 (Z - word 9) / word 9
//   distributions: far block [9, 10 + 3 nh): the monopole's third word, p, then the
//                  coefficients h, then l, then the third words of those after the
//                  monopole (nh = number of Hermite coefficients);
//                  L <= 2, near-capable tiles: general block of 2 + 2 nh words: sqrt(p) h, l,
//                  sqrt(pi)/2 G h, then l.
#pragma once

#include "esp_internal.h"

namespace esp {

constexpr int kDdGeneralMaxL = 2;         // larger L takes the FP64 code when not far
// The words of an offset hold it to 2^-48 q, and its hi word alone (the
// difference of two roundings to the grid q) is off by up to sqrt(3) q; q, 2^-24
// times a power of two above 4 max |P|, follows the farthest centre.  So words
// are used where offsets are long enough, which distant charges decide:
//  - at FP64 accuracy (three words): from 256 q on, so that the offset's error
//    is below 2^-56 of it and T = p |P - C|^2 from hi words within 1.4 %; in
//    environments with q up to kTdMaxQuantum (16,384 bohr), which also keeps d^4
//    below 2^64 (FP32's range);
//  - in 48 bits (beside FP32 sums): point charges from 4 q on, distributions of
//    q sqrt(p) <= 1; with q up to kDdMaxQuantum (a million bohr).
// The rest takes the FP64 code, as do point charges closer than 2^-10 bohr.
constexpr double kDdMaxQuantum = 0x1p-2, kTdMaxQuantum = 0x1p-8;
// T below which an entry is near (FP64): 45 where the asymptotic form holds to
// 1e-20, and a margin for T from the hi words
constexpr float kTdNearT = 46.0f;
constexpr float kDdMinR2 = 0x1p-20f;
// Smallest |P - C|^2 in words; lim = 2^23 q (dd_limit).  At most 1.
ESP_HD float dd_min_r2(float lim) { return fmaxf(kDdMinR2, (lim * 0x1p-21f) * (lim * 0x1p-21f)); }
ESP_HD float td_min_r2(float lim) { return fmaxf(kDdMinR2, (lim * 0x1p-15f) * (lim * 0x1p-15f)); }
// three words at all (by 2^23 q)
ESP_HD bool td_resolves(float lim) { return lim <= float(0x1p23 * kTdMaxQuantum); }
// Is an entry far, by T and |P - C|^2 from hi words?
ESP_HD bool td_is_far(float T, float r2, float min_r2) { return T >= kTdNearT && r2 >= 1.03f * min_r2; }
ESP_HD constexpr int dd_pad(int n) { return (n + 3) & ~3; }
constexpr int kDdPointWords = 13;
ESP_HD constexpr int dd_far_words(int L) { return 10 + 3 * num_hermite(L); }
ESP_HD constexpr int dd_gen_words(int L) { return L <= kDdGeneralMaxL ? 2 + 2 * num_hermite(L) : 0; }
// does a tile hold the general block (it can be near a position of an FP32C call)?
ESP_HD bool dd_has_general(const TileMeta &m)
{
    return m.cls <= kDdGeneralMaxL && m.vmax >= kNearVmax;
}
ESP_HD int dd_words(const TileMeta &m)
{
    if (is_point_class(m.cls))
        return kDdPointWords;
    return dd_far_words(m.cls & 7) + (dd_has_general(m) ? dd_gen_words(m.cls & 7) : 0);
}

// Boys table of the dd general form: rows at T_i = i / 64 up to 45, F_0..F_8 in
// units of sqrt(pi)/2 in FP32, then the low words of F_0..F_4, pad: 16 floats (one 64-byte line).
constexpr int kBoysDdRows = 45 * 64 + 2;
constexpr int kBoysDdRow = 16;
constexpr int kBoysDdHi = 9;
constexpr float kBoysDdTmax = 45.0f;

// one value per lane, h + l
struct dd {
    f2 h, l;
};

// a b = p + e exactly
ESP_HD f2 two_prod(f2 a, f2 b, f2 &e)
{
    const f2 p = a * b;
    e = esp_fma(a, b, -p);
    return p;
}
// a + b = s + e exactly (Knuth)
ESP_HD f2 two_sum(f2 a, f2 b, f2 &e)
{
    const f2 s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}
// the same for |a| >= |b| or a = 0 (Dekker)
ESP_HD f2 fast_two_sum(f2 a, f2 b, f2 &e)
{
    const f2 s = a + b;
    e = b - (s - a);
    return s;
}
ESP_HD dd dd_mul(dd a, dd b)
{
    f2 e;
    const f2 p = two_prod(a.h, b.h, e);
    return {p, esp_fma(a.l, b.h, esp_fma(a.h, b.l, e))};
}
ESP_HD dd dd_sqr(dd a)
{
    f2 e;
    const f2 p = two_prod(a.h, a.h, e);
    return {p, esp_fma(a.h + a.h, a.l, e)};
}
ESP_HD dd dd_add(dd a, dd b)
{
    f2 e;
    const f2 s = two_sum(a.h, b.h, e);
    return {s, (a.l + b.l) + e};
}
// |a| >= |b|
ESP_HD dd dd_add_small(dd a, dd b)
{
    f2 e;
    const f2 s = fast_two_sum(a.h, b.h, e);
    return {s, (a.l + b.l) + e};
}
ESP_HD dd dd_norm(dd a)
{
    f2 e;
    const f2 s = fast_two_sum(a.h, a.l, e);
    return {s, e};
}

// One coordinate of P - C from the three words of each.
ESP_HD dd dd_offset(f2 ph, f2 pm, f2 pl, float ch, float cm, float cl)
{
    f2 e;
    const f2 s = fast_two_sum(ph - f2(ch), pm - f2(cm), e);
    return {s, e + (pl - f2(cl))};
}

// x^2 + y^2 + z^2
ESP_HD dd dd_norm2(dd x, dd y, dd z)
{
    f2 ex, ey, ez, e1, e2;
    const f2 px = two_prod(x.h, x.h, ex), py = two_prod(y.h, y.h, ey), pz = two_prod(z.h, z.h, ez);
    const f2 s = two_sum(px, py, e1), r = two_sum(s, pz, e2);
    // Low part 2 h l + l^2 + the errors of the squares and sums.  An addition
    // drops low bits the same way in every term where they follow a pattern
    // (squares: 0, 1 or 4 modulo 8) or lie wholly below the other addend (l^2):
    // a shift of up to 1e-15 of every r^2.  Inside an FMA the product's bits
    // are as good as random, so l^2, ex and ey go there.
    const f2 u = esp_fma(x.l, x.l, esp_fma(y.l, y.l, z.l * z.l));
    const f2 tx = esp_fma(x.h + x.h, x.l, u), ty = esp_fma(y.h + y.h, y.l, ex), tz = esp_fma(z.h + z.h, z.l, ey);
    return dd_norm({r, ((tx + ty) + (tz + ez)) + (e1 + e2)});
}

// 1 / sqrt(a) as y (1 + u): y the FP32 value after one Newton step,
// u = -t/2 + 3/8 t^2 with the residual t = a y^2 - 1 (below 2^-23) in two parts:
// t1 = a.h p - 1 (exact but for its last bit or two) and s, the products with
// the low words.  rho is added to u: with the relative low word of a factor Z,
// Z.h y (1 + u) is Z / sqrt(a) with few roundings of the low part.
struct DdInv {
    f2 y, u;
};
ESP_HD DdInv dd_inv(dd a, f2 rho)
{
    const f2 y = esp_rsqrt(a.h);
    f2 e;
    const f2 p = two_prod(y, y, e);
    const f2 t1 = esp_fma(a.h, p, f2(-1.0f));
    const f2 s = esp_fma(a.h, e, a.l * p);
    const f2 t = t1 + s;
    return {y, esp_fma(0.375f * t, t, esp_fma(t1, f2(-0.5f), esp_fma(s, f2(-0.5f), rho)))};
}
ESP_HD dd dd_rsqrt(dd a)
{
    const DdInv v = dd_inv(a, f2(0.0f));
    return {v.y, v.y * v.u};
}
// z / sqrt(a) for z = zh (1 + rho)
ESP_HD dd dd_div_sqrt(f2 zh, f2 rho, dd a)
{
    const DdInv v = dd_inv(a, rho);
    f2 e;
    const f2 p = two_prod(zh, v.y, e);
    return {p, esp_fma(p, v.u, e)};
}

// Homogeneous polynomial of degree N with coefficients c(k), k the canonical
// index of the monomial among those of degree N (by descending power of x,
// then of y), by nested Horner schemes: x (x (..) + ..) + ...
template <int N, typename C>
ESP_HD dd dd_form(dd x, dd y, dd z, C c)
{
    if constexpr (N == 1) {
        return dd_add(dd_add(dd_mul(c(0), x), dd_mul(c(1), y)), dd_mul(c(2), z));
    } else {
        // the monomials with x (N (N + 1) / 2 of them) are x times a form of
        // degree N - 1; the rest is a form in y, z
        dd v = dd_mul(x, dd_form<N - 1>(x, y, z, c));
        constexpr int k0 = N * (N + 1) / 2;
        dd w = dd_add(dd_mul(c(k0), y), dd_mul(c(k0 + 1), z));
#pragma unroll
        for (int k = 2; k <= N; ++k) {
            // w y + c z^k, powers of z recomputed (N <= 4)
            dd zk = z;
            for (int i = 1; i < k; ++i)
                zk = dd_mul(zk, z);
            w = dd_add(dd_mul(w, y), dd_mul(c(k0 + k), zk));
        }
        return dd_add(v, w);
    }
}

// x = h + m + l as described above; returns the rest x - h.  (q is a power of
// two: the products with iq = 1 / q are exact.)
ESP_HD double dd_split3(double x, double q, double iq, float &h, float &m, float &l)
{
    const double qm = q * 0x1p-23;
    const double xh = nearbyint(x * iq) * q, r = x - xh, xm = nearbyint(r * (iq * 0x1p+23)) * qm;
    h = float(xh);
    m = float(xm);
    l = float(r - xm);
    return r;
}
ESP_HD void dd_split2(double x, float &h, float &l)
{
    h = float(x);
    l = float(x - double(h));
}

// x = h (1 + rho)
ESP_HD void dd_split_rel(double x, float &h, float &rho)
{
    h = float(x);
    rho = h != 0.0f ? float((x - double(h)) / double(h)) : 0.0f;
}

// (-1)^N (2N - 1)!! times the harmonic projection of the homogeneous
// polynomial c of degree N (canonical order), in place:
// P - r^2 lap P / (2 (2N - 1)) + r^4 lap^2 P / (8 (2N - 1)(2N - 3)), N <= 4.
template <int N>
ESP_HD void dd_project(double *c)
{
    constexpr double f = N == 1 ? -1.0 : N == 2 ? 3.0 : N == 3 ? -15.0 : 105.0;
    constexpr int off = N * (N + 1) * (N + 2) / 6;
    if constexpr (N >= 2) {
        constexpr int n2 = (N - 1) * N / 2, off2 = (N - 2) * (N - 1) * N / 6;
        double lap[6];
        for (int t = 0; t <= N - 2; ++t)
            for (int u = 0; t + u <= N - 2; ++u) {
                const int v = N - 2 - t - u;
                lap[hidx(t, u, v) - off2] = (t + 2) * (t + 1) * c[hidx(t + 2, u, v) - off] +
                                            (u + 2) * (u + 1) * c[hidx(t, u + 2, v) - off] +
                                            (v + 2) * (v + 1) * c[hidx(t, u, v + 2) - off];
            }
        // what is subtracted is r^2 times b = lap P / (2 (2N - 1)) - r^2 lap^2 P / (8 (2N - 1)(2N - 3))
        double b[6];
        for (int k = 0; k < n2; ++k)
            b[k] = lap[k] / (2.0 * (2 * N - 1));
        if constexpr (N == 4) {
            const double l2 = 2.0 * (lap[0] + lap[3] + lap[5]) / (8.0 * (2 * N - 1) * (2 * N - 3));
            b[0] -= l2;
            b[3] -= l2;
            b[5] -= l2;
        }
        for (int t = 0; t <= N - 2; ++t)
            for (int u = 0; t + u <= N - 2; ++u) {
                const int v = N - 2 - t - u;
                const double x = b[hidx(t, u, v) - off2];
                c[hidx(t + 2, u, v) - off] -= x;
                c[hidx(t, u + 2, v) - off] -= x;
                c[hidx(t, u, v + 2) - off] -= x;
            }
    }
    for (int k = 0; k < (N + 1) * (N + 2) / 2; ++k)
        c[k] *= f;
}

// The dd words of one FP64 record r of class cls, word w to out[w * n4].
template <int L>
ESP_HD void dd_convert_dist(const double *r, bool shortr, bool general, float *out, int n4)
{
    constexpr int nh = num_hermite(L);
    double M[nh];
    const double ip = 1.0 / r[3];
    double s = 0.88622692545275801365 * ip; // M_tuv = (pi / p)^{3/2} D_tuv = G_tuv sqrt(pi)/2 p^{-(N+1)/2}
    for (int N = 0, k = 0; N <= L; ++N, s *= ip)
        for (int e = 0; e < (N + 1) * (N + 2) / 2; ++e, ++k)
            M[k] = r[4 + k] * s;
    if (shortr)
        M[0] = 0.0;
    if constexpr (L >= 1)
        dd_project<1>(M + 1);
    if constexpr (L >= 2)
        dd_project<2>(M + 4);
    if constexpr (L >= 3)
        dd_project<3>(M + 10);
    if constexpr (L >= 4)
        dd_project<4>(M + 20);
    for (int k = 0; k < nh; ++k) {
        float &h = out[(11 + k) * n4], &l = out[(11 + nh + k) * n4];
        dd_split2(M[k], h, l);
        out[(k == 0 ? 9 : 10 + 2 * nh + k) * n4] = float(M[k] - double(h) - double(l));
    }
    out[10 * n4] = float(r[3] * r[3]);
    if (L <= kDdGeneralMaxL && general) {
        constexpr int go = dd_far_words(L);
        dd_split2(L == 0 ? r[3] * r[3] : r[3], out[go * n4], out[(go + 1) * n4]);
        for (int k = 0; k < nh; ++k)
            dd_split2(r[4 + k] * 0.88622692545275801365, out[(go + 2 + k) * n4], out[(go + 2 + nh + k) * n4]);
    }
}

ESP_HD void dd_convert(const TileMeta &m, const double *r, double q, float *out, int n4)
{
    const int cls = m.cls;
    const bool gen = dd_has_general(m);
    for (int d = 0; d < 3; ++d)
        dd_split3(r[d], q, 1.0 / q, out[d * n4], out[(3 + d) * n4], out[(6 + d) * n4]);
    const bool sh = (cls & kClassShortBit) != 0;
    if (is_point_class(cls)) {
        float h, rho, l;
        dd_split_rel(r[3], h, rho);
        dd_split2(r[3], h, l);
        out[9 * n4] = h;
        out[10 * n4] = l;
        out[11 * n4] = float(r[3] - double(h) - double(l));
        out[12 * n4] = rho;
        return;
    }
    switch (cls & 7) {
    case 0: dd_convert_dist<0>(r, sh, gen, out, n4); break;
    case 1: dd_convert_dist<1>(r, sh, gen, out, n4); break;
    case 2: dd_convert_dist<2>(r, sh, gen, out, n4); break;
    case 3: dd_convert_dist<3>(r, sh, gen, out, n4); break;
    default: dd_convert_dist<4>(r, sh, gen, out, n4); break;
    }
}

// ---------------------------------------------------------------------------
// The far form at FP64 accuracy.  One rounding of a low word costs up to
// 2^-49 of the result, and the dd form above makes about fifteen of them
// (3e-15 rms per term, against 1e-16 of FP64 arithmetic, which many-term sums
// average but small ones show).  Here r^2 = a + b + c has a third word and the
// roundings of the second are kept in it; the residual of the reciprocal
// square root is summed from exact products.
// ---------------------------------------------------------------------------
struct Td {
    f2 a, b, c;
};
// Three words a + b + c that need not be normalised: |b| up to a few 2^-23 |a|,
// c the rest in FP32.  A product or sum keeps every rounding of the first two
// words, so its error is that of c: below 2^-60 of the operands' size.
ESP_HD Td td_mul(const Td &x, const Td &y)
{
    f2 e, f, g, e1, e2;
    const f2 p = two_prod(x.a, y.a, e), q = two_prod(x.a, y.b, f), r = two_prod(x.b, y.a, g);
    f2 b = two_sum(q, r, e1);
    b = two_sum(b, e, e2);
    return {p, b, esp_fma(x.b, y.b, esp_fma(x.a, y.c, esp_fma(x.c, y.a, f + g))) + (e1 + e2)};
}
ESP_HD Td td_sqr(const Td &x)
{
    f2 e, f, e1;
    const f2 p = two_prod(x.a, x.a, e), q = two_prod(x.a + x.a, x.b, f);
    const f2 b = two_sum(q, e, e1);
    return {p, b, esp_fma(x.b, x.b, esp_fma(x.a + x.a, x.c, f + e1))};
}
ESP_HD Td td_add(const Td &x, const Td &y)
{
    f2 e, e1, e2;
    const f2 a = two_sum(x.a, y.a, e);
    f2 b = two_sum(x.b, y.b, e1);
    b = two_sum(b, e, e2);
    return {a, b, (x.c + y.c) + (e1 + e2)};
}
// dd_form in three words
template <int N, typename C>
ESP_HD Td td_form(const Td &x, const Td &y, const Td &z, C c)
{
    if constexpr (N == 1) {
        return td_add(td_add(td_mul(c(0), x), td_mul(c(1), y)), td_mul(c(2), z));
    } else {
        const Td v = td_mul(x, td_form<N - 1>(x, y, z, c));
        constexpr int k0 = N * (N + 1) / 2;
        Td w = td_add(td_mul(c(k0), y), td_mul(c(k0 + 1), z));
        Td zk = z;
#pragma unroll
        for (int k = 2; k <= N; ++k) {
            zk = k == 2 ? td_sqr(z) : td_mul(zk, z);
            w = td_add(td_mul(w, y), td_mul(c(k0 + k), zk));
        }
        return td_add(v, w);
    }
}
// offset in three words: s + e exactly h + m, l the rest
struct TdOff {
    f2 s, e, l;
};
ESP_HD TdOff td_offset(f2 ph, f2 pm, f2 pl, float ch, float cm, float cl)
{
    TdOff o;
    o.s = fast_two_sum(ph - f2(ch), pm - f2(cm), o.e);
    o.l = pl - f2(cl);
    return o;
}
// b += x with the rounding error added to c
ESP_HD void td_acc(f2 &b, f2 &c, f2 x)
{
    f2 e;
    b = two_sum(b, x, e);
    c += e;
}
ESP_HD Td td_norm2(const TdOff &x, const TdOff &y, const TdOff &z)
{
    f2 ex, ey, ez, e1, e2, fx, fy, fz, e;
    const f2 px = two_prod(x.s, x.s, ex), py = two_prod(y.s, y.s, ey), pz = two_prod(z.s, z.s, ez);
    const f2 x2 = x.s + x.s, y2 = y.s + y.s, z2 = z.s + z.s;
    const f2 qx = two_prod(x2, x.e, fx), qy = two_prod(y2, y.e, fy), qz = two_prod(z2, z.e, fz);
    f2 a = two_sum(px, py, e1);
    a = two_sum(a, pz, e2);
    f2 c = esp_fma(x2, x.l, esp_fma(x.e, x.e, fx)) +
           (esp_fma(y2, y.l, esp_fma(y.e, y.e, fy)) + esp_fma(z2, z.l, esp_fma(z.e, z.e, fz)));
    f2 b = qx;
    td_acc(b, c, qy);
    td_acc(b, c, qz);
    td_acc(b, c, ex);
    td_acc(b, c, ey);
    td_acc(b, c, ez);
    td_acc(b, c, e1);
    td_acc(b, c, e2);
    a = fast_two_sum(a, b, e);
    return {a, e, c};
}
// Sum of three-word values over a few records: a the leading products, b what
// lies about 2^-24 below, c the roundings of both.
struct TdSum {
    f2 a, b, c;
    ESP_HD void clear() { a = b = c = f2(0.0f); }
    ESP_HD void mid(f2 x) { td_acc(b, c, x); }
    // add z / sqrt(r2) for z = zh + zl + zm; returns 1 / sqrt(r2)
    ESP_HD Td div_sqrt(f2 zh, f2 zl, f2 zm, const Td &r2)
    {
        const f2 y = esp_rsqrt(r2.a);
        f2 pe, qe, fe, ge, he, ze, ke, le, e;
        const f2 p = two_prod(y, y, pe);
        const f2 q = two_prod(r2.a, p, qe);
        const f2 t1 = q - f2(1.0f); // exact
        // t = r2 y^2 - 1 = t1 + mid + low
        const f2 f = two_prod(r2.a, pe, fe), g = two_prod(r2.b, p, ge);
        f2 low = esp_fma(r2.b, pe, esp_fma(r2.c, p, fe + ge)), md = qe;
        td_acc(md, low, f);
        td_acc(md, low, g);
        // 1 / sqrt = y (1 - t/2 + 3/8 t^2)
        const f2 t = t1 + md;
        const f2 u3 = esp_fma(0.375f * t, t, -0.5f * low);
        const f2 u1 = -0.5f * t1, u2 = -0.5f * md;
        const f2 v = two_prod(zh, y, ze);
        const f2 h = two_prod(v, u1, he), k = two_prod(v, u2, ke), l = two_prod(zl, y, le);
        a = two_sum(a, v, e);
        mid(e);
        mid(h);
        mid(k);
        mid(l);
        mid(ze);
        const f2 u = u1 + u2;
        c += esp_fma(v, u3, esp_fma(l + ze, u, esp_fma(zm, y, (he + ke) + le)));
        f2 e1, e2, ye;
        const f2 y1 = two_prod(y, u1, e1), y2 = two_prod(y, u2, e2), yb = two_sum(y1, y2, ye);
        return {y, yb, esp_fma(y, u3, (e1 + e2) + ye)};
    }
    ESP_HD void add(const Td &x)
    {
        f2 e;
        a = two_sum(a, x.a, e);
        mid(e);
        mid(x.b);
        c += x.c;
    }
    ESP_HD double total() const
    {
        return ((double)a.x + (double)a.y) + (((double)b.x + (double)b.y) + (double)(c.x + c.y));
    }
};

// padding records: zero every coefficient (the exponent words stay)
ESP_HD void dd_zero_coefficients(const TileMeta &m, float *out, int n4)
{
    const int far_end = is_point_class(m.cls) ? kDdPointWords : dd_far_words(m.cls & 7);
    for (int w = 9; w < dd_words(m); ++w)
        if (is_point_class(m.cls) || (w != 10 && w != far_end && w != far_end + 1))
            out[w * n4] = 0.0f;
}

// Accessor of a dd tile: word w of records j, j + 1 (j even).
struct DdTile {
    const float *p;
    int n4;
    ESP_HD f2 operator()(int w, int j) const
    {
#if defined(__CUDA_ARCH__)
        const float2 v = *reinterpret_cast<const float2 *>(p + w * n4 + j);
        return f2(v.x, v.y);
#else
        return f2(p[w * n4 + j], p[w * n4 + j + 1]);
#endif
    }
};

// the nine words of a position: h, m, l of x, y, z
struct DdPos {
    float h[3], m[3], l[3];
};

ESP_HD void dd_offsets(const DdTile &t, int j, const DdPos &c, dd (&d)[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k)
        d[k] = dd_offset(t(k, j), t(3 + k, j), t(6 + k, j), c.h[k], c.m[k], c.l[k]);
}

// Point charges j, j + 1: Z / |P - C|; r2 receives |P - C|^2 (the caller
// re-evaluates in FP64 below dd_min_r2).
ESP_HD dd dd_point(const DdTile &t, int j, const DdPos &c, f2 &r2)
{
    dd d[3];
    dd_offsets(t, j, c, d);
    const dd s = dd_norm2(d[0], d[1], d[2]);
    r2 = s.h;
    return dd_div_sqrt(t(9, j), t(12, j), s);
}

// Far form of distributions j, j + 1 at FP64 accuracy, added to sum: every
// order in three words.  (The orders above the monopole in 48 bits, as they
// were, erred by up to 7e-15 of the terms, against 6e-16 of the FP64 code: they
// fall off as (size / distance)^N, but a product of s and p on one centre, say,
// has no monopole beside them.)  Lanes with use = 0 add nothing, whatever their offset; r2 receives
// |P - C|^2 (1 for those).
template <int L>
ESP_HD void td_far(const DdTile &t, int j, const DdPos &c, bool use0, bool use1, TdSum &sum, f2 &r2)
{
    constexpr int nh = num_hermite(L);
    TdOff o[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        o[k] = td_offset(t(k, j), t(3 + k, j), t(6 + k, j), c.h[k], c.m[k], c.l[k]);
    Td s = td_norm2(o[0], o[1], o[2]);
    s.a = f2(use0 ? s.a.x : 1.0f, use1 ? s.a.y : 1.0f);
    s.b = f2(use0 ? s.b.x : 0.0f, use1 ? s.b.y : 0.0f);
    s.c = f2(use0 ? s.c.x : 0.0f, use1 ? s.c.y : 0.0f);
    r2 = s.a;
    const f2 w(use0 ? 1.0f : 0.0f, use1 ? 1.0f : 0.0f);
    const Td y = sum.div_sqrt(w * t(11, j), w * t(11 + nh, j), w * t(9, j), s);
    if constexpr (L > 0) {
        auto coef = [&](int k) { return Td{t(11 + k, j), t(11 + nh + k, j), t(10 + 2 * nh + k, j)}; };
        const Td x = {o[0].s, o[0].e, o[0].l}, yy = {o[1].s, o[1].e, o[1].l}, z = {o[2].s, o[2].e, o[2].l};
        const Td i2 = td_sqr(y);
        // Horner's scheme in 1 / r^2 from the highest order down
        Td v = td_form<L>(x, yy, z, [&](int k) { return coef(L * (L + 1) * (L + 2) / 6 + k); });
        if constexpr (L >= 4)
            v = td_add(td_form<3>(x, yy, z, [&](int k) { return coef(10 + k); }), td_mul(i2, v));
        if constexpr (L >= 3)
            v = td_add(td_form<2>(x, yy, z, [&](int k) { return coef(4 + k); }), td_mul(i2, v));
        if constexpr (L >= 2)
            v = td_add(td_form<1>(x, yy, z, [&](int k) { return coef(1 + k); }), td_mul(i2, v));
        v = td_mul(td_mul(i2, y), v);
        sum.add(Td{w * v.a, w * v.b, w * v.c});
    }
}
// Point charges j, j + 1 at FP64 accuracy.
ESP_HD void td_point(const DdTile &t, int j, const DdPos &c, TdSum &sum, f2 &r2)
{
    TdOff o[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        o[k] = td_offset(t(k, j), t(3 + k, j), t(6 + k, j), c.h[k], c.m[k], c.l[k]);
    const Td s = td_norm2(o[0], o[1], o[2]);
    r2 = s.a;
    sum.div_sqrt(t(9, j), t(10, j), t(11, j), s);
}

// F_0..F_L of one lane's T (h + l, below kBoysDdTmax) from the table: Taylor
// about T_i = i / 64 (|T - T_i| <= 1/128: the terms beyond the sixth are below
// 2^-54, those beyond the second need FP32 only).
template <int L>
ESP_HD void boys_dd(float Th, float Tl, const float *__restrict__ tab, float (&Fh)[L + 1], float (&Fl)[L + 1])
{
    const int i = (int)(Th * 64.0f + 0.5f);
    const float *row = tab + i * kBoysDdRow;
    const float mh = float(i) * 0.015625f - Th; // -(T - T_i), exact
    const float mh3 = mh * (1.0f / 3.0f), mh4 = mh * 0.25f, mh5 = mh * 0.2f, mh6 = mh * (1.0f / 6.0f);
    const float hh = 0.5f * mh, hl = -0.5f * Tl;
    float F[kBoysDdHi], G[5];
#if defined(__CUDA_ARCH__)
    {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
        const float4 a = __ldg(r4), b = __ldg(r4 + 1), c = __ldg(r4 + 2), d = __ldg(r4 + 3);
        F[0] = a.x, F[1] = a.y, F[2] = a.z, F[3] = a.w, F[4] = b.x, F[5] = b.y, F[6] = b.z, F[7] = b.w, F[8] = c.x;
        G[0] = c.y, G[1] = c.z, G[2] = c.w, G[3] = d.x, G[4] = d.y;
    }
#else
    for (int k = 0; k < kBoysDdHi; ++k)
        F[k] = row[k];
    for (int k = 0; k < 5; ++k)
        G[k] = row[kBoysDdHi + k];
#endif
#pragma unroll
    for (int n = 0; n <= L; ++n) {
        float f = fmaf(F[n + 6], mh6, F[n + 5]);
        f = fmaf(f, mh5, F[n + 4]);
        f = fmaf(f, mh4, F[n + 3]);
        const float a = f * mh3;
        float sh = F[n + 2] + a, sl = G[n + 2] + (a - (sh - F[n + 2]));
#pragma unroll
        for (int k = 1; k >= 0; --k) { // times (mh, -Tl) / (2 - k + ... ): halves first, then whole
            const float xh = k ? hh : mh, xl = k ? hl : -Tl;
            const float p = sh * xh;
            const float e = fmaf(sl, xh, fmaf(sh, xl, fmaf(sh, xh, -p)));
            sh = F[n + k] + p;
            sl = (G[n + k] + e) + (p - (sh - F[n + k]));
        }
        Fh[n] = sh;
        Fl[n] = sl;
    }
}

// General form of distributions j, j + 1 (L <= 2, not the short-range kind,
// whose difference from the monopole needs FP64).  go: word of the general
// block; for L = 0 also reads the far block (words 11, 12).
template <int L>
ESP_HD dd dd_general(const DdTile &t, int j, const DdPos &c, int go, const float *__restrict__ tab)
{
    static_assert(L <= kDdGeneralMaxL, "no dd general form");
    constexpr int nh = num_hermite(L);
    dd x[3];
    dd_offsets(t, j, c, x);
    const dd sp = {t(go, j), t(go + 1, j)}; // L = 0: p
    auto G = [&](int k) { return dd{t(go + 2 + k, j), t(go + 2 + nh + k, j)}; };
    if constexpr (L == 0) {
        const dd r2 = dd_norm2(x[0], x[1], x[2]);
        dd v = dd_mul({t(11, j), t(12, j)}, dd_rsqrt(r2)); // asymptotic form
        const dd T = dd_norm(dd_mul(sp, r2));
        const bool a0 = T.h.x >= kBoysDdTmax, a1 = T.h.y >= kBoysDdTmax;
        if (!(a0 && a1)) {
            dd F = {f2(0.0f), f2(0.0f)};
            float fh[1], fl[1];
            if (!a0) {
                boys_dd<0>(T.h.x, T.l.x, tab, fh, fl);
                F.h.x = fh[0], F.l.x = fl[0];
            }
            if (!a1) {
                boys_dd<0>(T.h.y, T.l.y, tab, fh, fl);
                F.h.y = fh[0], F.l.y = fl[0];
            }
            const dd w = dd_mul(G(0), F);
            v.h = f2(a0 ? v.h.x : w.h.x, a1 ? v.h.y : w.h.y);
            v.l = f2(a0 ? v.l.x : w.l.x, a1 ? v.l.y : w.l.y);
        }
        return v;
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k)
            x[k] = dd_norm(dd_mul(sp, x[k]));
        const dd T = dd_norm(dd_norm2(x[0], x[1], x[2]));
        // asymptotic: F_0 = 1 / sqrt(T), F_n = F_{n-1} (2n - 1) / (2T) (Boys
        // values in units of sqrt(pi)/2 here, which the coefficients carry: a
        // constant rounded to 48 bits would shift every term the same way)
        const dd y = dd_rsqrt(T);
        dd F[L + 1];
        F[0] = y;
        const bool a0 = T.h.x >= kBoysDdTmax, a1 = T.h.y >= kBoysDdTmax;
        const dd i2 = dd_sqr(y); // 1 / T
        const dd h = {0.5f * i2.h, 0.5f * i2.l};
        F[1] = dd_mul(F[0], h);
        if constexpr (L > 1) {
            const dd t3 = dd_mul(F[1], h);
            F[2] = dd_add_small({t3.h + t3.h, t3.l + t3.l}, t3); // 3 t: 2 t + t with its rounding kept
        }
        if (!a0) {
            float fh[L + 1], fl[L + 1];
            boys_dd<L>(T.h.x, T.l.x, tab, fh, fl);
#pragma unroll
            for (int n = 0; n <= L; ++n)
                F[n].h.x = fh[n], F[n].l.x = fl[n];
        }
        if (!a1) {
            float fh[L + 1], fl[L + 1];
            boys_dd<L>(T.h.y, T.l.y, tab, fh, fl);
#pragma unroll
            for (int n = 0; n <= L; ++n)
                F[n].h.y = fh[n], F[n].l.y = fl[n];
        }
        // sum over orders with the traces collected per Boys value
        dd a = dd_form<1>(x[0], x[1], x[2], [&](int k) { return G(1 + k); });
        if constexpr (L > 1)
            a = dd_add(a, dd_add(dd_add(G(4), G(7)), G(9))); // x^2, y^2, z^2
        a = dd_mul(a, F[1]);
        dd v = dd_add(dd_mul(G(0), F[0]), {-(a.h + a.h), -(a.l + a.l)});
        if constexpr (L > 1) {
            const dd b = dd_mul(dd_form<2>(x[0], x[1], x[2], [&](int k) { return G(4 + k); }), F[2]);
            v = dd_add(v, {4.0f * b.h, 4.0f * b.l});
        }
        return v;
    }
}

} // namespace esp
