// Host check of the sweeps' fixed-point arithmetic (csrc/fixed.cuh) against long double: prints, per part,
// the largest error over its bound. usage: fixed_point_check exp | scaled | conv | sums N order
#include "fixed.cuh"

#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

using namespace kitrt_fx;
typedef long double LD;
const LD kPi = 3.14159265358979323846264338327950288L;

std::vector<uint64_t> exp_table()
{
    std::vector<uint64_t> t(2048);
    for (int j = 0; j < 2048; ++j) t[j] = (uint64_t)llroundl(exp2l(61.0L + j / 2048.0L));
    return t;
}

// 2^(s / 2048), s in units of 2^-42: relative error over 2^-51
double check_exp()
{
    const auto tab = exp_table();
    std::mt19937_64 g(1);
    LD worst = 0;
    for (int i = 0; i < 2000000; ++i) {
        long long s = (long long)g() >> (2 + g() % 40);  // below 2^61.5 in magnitude, every size
        if (i % 8 == 0) s = (s >> 42 << 42) - (i & 8 ? 1 : 0);  // both ends of a table interval
        const Exp e = fx_exp(s, tab.data());
        const LD want = exp2l(ldexpl((LD)(s & ((1LL << 53) - 1)), -53));  // 2^fraction, exponent s >> 53
        const LD got = ldexpl((LD)e.y, -61 + e.m - (int)(s >> 53));
        worst = std::max(worst, fabsl(got / want - 1));
    }
    return (double)(worst * ldexpl(1, 51));
}

// 2^(s 2^sh / 2048) of scaled rows: relative error over 2^-51; 2^-1024 at -707 and below, refused beyond a double
double check_scaled()
{
    const auto tab = exp_table();
    std::mt19937_64 g(3);
    LD worst = 0;
    for (int i = 0; i < 2000000; ++i) {
        const int sh = 1 + (int)(g() % kMaxShift);
        // z in +-800, or of any size that the row's range has
        const LD z = ((LD)(long long)g() / 9223372036854775808.0L) * (i % 4 ? 800.0L : ldexpl(128, sh));
        const long long s = llroundl(ldexpl(z * 2048 / logl(2), kFracBits - sh));
        const LD x = ldexpl((LD)s, sh - 53);  // log2 of the value
        long long full = s;
        const bool in = fx_unscale(full, sh);
        const Exp e = fx_exp(full, tab.data());
        if (x * logl(2) < -707.001L) worst = std::max(worst, (LD)(in && e.m == -1024 ? 0 : 1e9));
        else if (x >= 1024) worst = std::max(worst, (LD)(!in && e.m == 1023 ? 0 : 1e9));
        else if (x * logl(2) > -706.999L) worst = std::max(worst, in ? fabsl(ldexpl((LD)e.y, e.m - 61) / exp2l(x) - 1) : 1e9L);
    }
    for (double z : {0.0, -1e-300, -706.99, 1.0, -3.25, 700.0, 709.7}) {
        long long s;
        const bool in = fx_exponent_of(z, s);
        // the exponent rounded twice to 53 bits
        const LD tol = ldexpl(1, -51) + ldexpl(fabs(z), -51);
        const Exp e = fx_exp(s, tab.data());
        worst = std::max(worst, in ? fabsl(ldexpl((LD)e.y, e.m - 61) / expl(z) - 1) / tol * ldexpl(1, -51) : 1e9L);
    }
    for (double z : {709.79, (double)INFINITY, (double)NAN, -707.0, -1e300, (double)-INFINITY}) {
        long long s;
        if (fx_exponent_of(z, s) != (z < 0) || s != (z < 0 ? INT64_MIN : INT64_MAX)) worst = 1e9;
    }
    for (float b : {0.0f, 244.99f, 245.0f, 256.0f, 1e4f, 1e11f, 5e11f}) {
        const int sh = fx_row_shift(b);
        if (sh < 0 || !(ldexpf(b, -sh) < (sh ? 128.0f : 245.0f))) worst = 1e9;
    }
    for (float b : {1e13f, INFINITY, NAN})
        if (fx_row_shift(b) != -1) worst = 1e9;
    return (double)(worst * ldexpl(1, 51));
}

// conversions, exact up to their rounding (half a unit of the result)
double check_conv()
{
    std::mt19937_64 g(2);
    LD worst = 0;
    for (int i = 0; i < 1000000; ++i) {
        const double x = ldexp((double)(long long)g(), -63) * ldexp(1.0, (int)(g() % 80) - 70);
        worst = std::max(worst, fabsl((LD)fx_from_double(x) - ldexpl((LD)x, 52)) * 2);
        const int down = (int)(g() % 33);
        worst = std::max(worst, fabsl((LD)fx_from_double(x, down) - ldexpl((LD)x, 52 - down)) * 2);
        const long long v = (long long)g() >> (g() % 64);
        const int sh = (int)(g() % 200) - 100;
        const double d = fx_to_double(v, sh);
        const LD unit = v ? ldexpl(1, std::max(0, 64 - 53 - __builtin_clzll(v < 0 ? -(unsigned long long)v : v)) + sh) : 1;
        worst = std::max(worst, fabsl((LD)d - ldexpl((LD)v, sh)) / unit * 2);
    }
    return (double)worst;
}

// Moments of one pass over the rule, degree 2N, against the sums of the same (rounded) exponentials and tables.
// In units of the sums: an exponential e is rounded by at most min(e, 1/2), a quad's dropped low
// product is at most min(c, 2^26) 2^-28 (c: the quad's combination), each azimuthal sum is rounded by
// 1/2, each ring's term of a moment by 2^sh / 2; when the scale rises, each sum loses up to 1. These
// are independent and without bias, so that the bound is six standard deviations (each at most its
// largest value over sqrt 3) of their sum: a bias of a fraction of a unit per point fails it.
template <int N>
double check_sums(int order)
{
    constexpr int n = (N + 1) * (N + 2) / 2, L2 = 2 * N, n2 = (L2 + 1) * (L2 + 2) / 2;
    const int P = order, J = (P + 1) / 2, R = order / 2 + order % 2;
    std::vector<double> Pn((size_t)R * n2), w(R);
    for (int r = 0; r < R; ++r) {
        LD x = cosl(kPi * (r + 0.75L) / (order + 0.5L)), dp = 1;
        const bool mid = order % 2 && r == R - 1;
        if (mid) x = 0;
        for (int it = 0; it < 60; ++it) {
            LD a = 1, b = x;
            for (int j = 2; j <= order; ++j) {
                const LD c = ((2 * j - 1) * x * b - (j - 1) * a) / j;
                a = b;
                b = c;
            }
            dp = order * (a - x * b) / (1 - x * x);
            if (!mid) x -= b / dp;
        }
        w[r] = (double)((mid ? 1 : 2) * 2 / ((1 - x * x) * dp * dp) * kPi / order);
        LD q[2 * N + 1][2 * N + 1] = {}, s = sqrtl(1 - x * x);
        q[0][0] = sqrtl(1 / (4 * kPi));
        for (int k = 1; k <= L2; ++k) q[k][k] = sqrtl((2 * k + 1.0L) / (2 * k)) * s * q[k - 1][k - 1];
        for (int k = 0; k < L2; ++k) q[k + 1][k] = sqrtl(2 * k + 3.0L) * x * q[k][k];
        for (int k = 0; k <= L2; ++k)
            for (int l = k + 2; l <= L2; ++l) {
                const LD a = sqrtl((4.0L * l * l - 1) / (l * l - k * k));
                const LD b = sqrtl(((l - 1.0L) * (l - 1) - k * k) / (4.0L * (l - 1) * (l - 1) - 1));
                q[l][k] = a * (x * q[l - 1][k] - b * q[l - 2][k]);
            }
        for (int l = 0; l <= L2; ++l)
            for (int k = -l; k <= l; k += 2) Pn[(size_t)r * n2 + cindex(l, k)] = (double)(q[l][abs(k)] * (k ? sqrtl(2) : 1));
    }
    // tables and units as kitrt_mn_init forms them
    double wmax = 0, most = 0;
    for (int c = 0; c < n2; ++c) {
        double sum = 0;
        for (int r = 0; r < R; ++r) {
            wmax = std::max(wmax, fabs(w[r] * Pn[(size_t)r * n2 + c]));
            sum += 2.0 * P * fabs(w[r] * Pn[(size_t)r * n2 + c]);
        }
        most = std::max(most, sum);
    }
    int wexp, sh;
    frexp(wmax, &wexp);
    frexp(ldexp(1.001 * most, -wexp), &sh);
    sh -= kGuard + 1;
    if (sh > 2) {
        wexp += sh - 2;
        sh = 2;
    }
    auto limbs = [](LD x, int bits) {
        const Limb l = split<27>(llroundl(ldexpl(x, bits)));
        int2 v;
        v.x = l.h;
        v.y = l.l;
        return v;
    };
    auto value = [](int2 v, int bits) { return ldexpl((LD)(((long long)v.x << 27) + v.y), -bits); };
    std::vector<int2> trig((size_t)J * 2 * L2), rA((size_t)R * n), rW((size_t)R * n2);
    for (int j = 0; j < J; ++j)
        for (int k = 1; k <= L2; ++k) {
            trig[(size_t)j * 2 * L2 + k - 1] = limbs(cosl(k * j * kPi / P), 54);
            trig[(size_t)j * 2 * L2 + L2 + k - 1] = limbs(sinl(k * j * kPi / P), 54);
        }
    for (int r = 0; r < R; ++r)
        for (int c = 0; c < n2; ++c) {
            if (c < n) rA[(size_t)r * n + c] = limbs((LD)Pn[(size_t)r * n2 + c] * 2048 / logl(2), 45);
            rW[(size_t)r * n2 + c] = limbs(ldexpl((LD)w[r] * Pn[(size_t)r * n2 + c], -wexp), 57);
        }
    const auto tab = exp_table();
    std::mt19937_64 g(order + 100 * N);
    std::normal_distribution<double> normal;
    LD worst = 0;
    for (int row = 0; row < 60; ++row) {
        // flat rows, and peaks of every sharpness: towards a pole (where the weights are small), in the plane
        double al[n];
        const double size = row % 4 ? exp(normal(g) + 3.0) : 0.5;
        for (int c = 0; c < n; ++c) al[c] = 0.3 * normal(g) * (row % 4 ? 1 : size);
        if (row % 4 == 1) al[cindex(N >= 2 ? 2 : 1, N >= 2 ? 0 : 1)] += size;
        if (row % 4 == 2) al[cindex(1, 1)] += size;
        al[0] = 10.0 * normal(g);
        Limb at[n];
        for (int c = 0; c < n; ++c) at[c] = split<32>(fx_from_double(al[c]));
        long long A0, V[n2] = {};
        Limb A[2 * N];
        FxSums<L2> B;
        B.clear();
        std::vector<Exp> all((size_t)R * J * 4);
        int raises = 0;
        for (int pass = 0; pass < 2; ++pass) {
            LD v0 = 0;
            for (int r = 0; r < R; ++r) {
                fx_coeffs<N>([&](int c) { return at[c]; }, &rA[(size_t)r * n], A0, A);
                for (int j = 0; j < J; ++j) {
                    long long s[4];
                    Exp *e = &all[4 * ((size_t)r * J + j)], q[4];
                    fx_exponents<N>(A0, A, &trig[(size_t)j * 2 * L2], L2, j == 0, s);
                    for (int t = 0; t < 4; ++t) e[t] = fx_exp(s[t], tab.data());
                    if (j == 0 && P % 2) e[2] = e[3] = Exp{0, -100000};
                    for (int t = 0; t < 4; ++t) {
                        q[t] = e[t];
                        if (q[t].y) v0 += ldexpl((LD)q[t].y, q[t].m - 61) * w[r] * Pn[(size_t)r * n2];
                    }
                    if (pass)
                        fx_accumulate<L2>(q, &trig[(size_t)j * 2 * L2], L2, j == 0, r + j == 0, B, [&](int d) {
                            ++raises;
                            for (auto &x : V) x = sar(x, d);
                        });
                }
                if (pass)
                    fx_flush<L2>(&rW[(size_t)r * n2], sh, B, [&](int c) -> long long & { return V[c]; });
            }
            if (!pass) B.Sx = fx_scale_of((double)v0);  // as a closure of its own moments
        }
        for (int l = 0; l <= L2; ++l)
            for (int k = -l; k <= l; k += 2) {
                const int c = cindex(l, k), ak = abs(k);
                LD ref = 0, var = raises * ldexpl(1.0L, 2 * sh);  // 3 x variance
                for (int r = 0; r < R; ++r) {
                    LD b = 0, vb = k ? 0.25L : 0;
                    for (int j = 0; j < J; ++j) {
                        LD T[4], c4 = 0;
                        if (j) {
                            const int2 *t = &trig[(size_t)j * 2 * L2];
                            const LD v = k == 0 ? 1 : k > 0 ? value(t[k - 1], 54) : value(t[L2 + ak - 1], 54);
                            const LD s = ak % 2 ? -1 : 1;  // phi, -phi, pi - phi, pi + phi
                            T[0] = v;
                            T[1] = k >= 0 ? v : -v;
                            T[2] = k >= 0 ? s * v : -s * v;
                            T[3] = s * v;
                        } else {
                            const LD s = ak % 2 ? -1 : 1, half = ak % 4 < 2 ? 1 : -1;
                            T[0] = k >= 0 ? 1 : 0;
                            T[1] = k >= 0 ? s : 0;
                            T[2] = k >= 0 ? (ak % 2 ? 0 : half) : (ak % 2 ? half : 0);
                            T[3] = k >= 0 ? T[2] : -T[2];
                        }
                        for (int t = 0; t < 4; ++t) {
                            const Exp e = all[4 * ((size_t)r * J + j) + t];
                            const LD f = e.y ? ldexpl((LD)e.y, e.m - B.Sx) : 0;
                            b += f * T[t];
                            c4 += f;
                            vb += T[t] * T[t] * std::min(f, 0.5L) * std::min(f, 0.5L);
                        }
                        const LD low = ldexpl(std::min(c4, ldexpl(1, 26)), -28);
                        if (j && k) vb += low * low;
                    }
                    const LD wp = value(rW[(size_t)r * n2 + c], 57);
                    ref += b * wp;
                    var += (vb + 1.0L * raises) * wp * wp + ldexpl(0.25L, 2 * sh);
                }
                worst = std::max(worst, fabsl(ldexpl((LD)V[c], sh) - ref) / (6 * sqrtl(var / 3)));
            }
    }
    return (double)worst;
}

int main(int argc, char **argv)
{
    const char *what = argc > 1 ? argv[1] : "";
    double r = 1e9;
    if (!strcmp(what, "exp")) r = check_exp();
    if (!strcmp(what, "scaled")) r = check_scaled();
    if (!strcmp(what, "conv")) r = check_conv();
    if (!strcmp(what, "sums") && argc > 3) {
        const int N = atoi(argv[2]), order = atoi(argv[3]);
        r = N == 1 ? check_sums<1>(order) : N == 2 ? check_sums<2>(order) : N == 3 ? check_sums<3>(order)
            : N == 4 ? check_sums<4>(order) : check_sums<5>(order);
    }
    printf("%.6f\n", r);
    return 0;
}
