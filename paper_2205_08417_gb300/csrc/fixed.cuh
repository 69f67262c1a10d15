// The quadrature sums of the closure's dual in 64-bit fixed point, on the integer pipes.
//
// FP64 runs at 2 lanes per clock per SM on this GPU (a warp instruction holds the pipe for 16
// cycles), 32-bit integer multiply-adds with a 64-bit result at 64 lanes. The sum-factorised pass
// of sweep.cuh (exponent coefficients per ring, exponentials per pair of mirrored azimuths,
// azimuthal sums per ring) needs nothing that a fixed binary point cannot hold, so every step is
// done in products of two-limb integers here (high and balanced low part): of the four partial
// products the low one is dropped, which costs at most 4 units of the result and has no bias.
// Formats:
//   exponent s = (alpha . m) 2048 / ln2 in units of 2^-42 (2^-53.5 of alpha . m), |s| < 2^61.5: rows
//   with sum_c |alpha_c| max|m_c| >= kFxMaxZ are scaled down by a power of two (fx_row_shift), which
//   leaves them at least 2^8 units per rounding error of an FP64 sum of that size;
//   azimuthal factors cos(k phi), sin(k phi) in units of 2^-54, the weighted Legendre factors of
//   the moments in units of 2^-57 of a power of two, the exponent's in units of 2^-45;
//   exponential e = y 2^(m - 61), y in [2^61, 2^62]: T_j (1 + p) with the 2048-entry table and
//   p = exp(r ln2/2048) - 1 on r in [0, 1) by a cubic whose quartic term is folded in (error below
//   2^-57); |error| of y below 2^-51 relative;
//   sums in units of 2^(Sx - 61): e is shifted down by Sx - m >= 7, so that it stays below 2^55 and
//   32 quads fit; Sx belongs to the row and is raised (and the sums shifted) when a larger
//   exponential appears. Exponentials are rounded to nearest: one far below the row's largest adds no
//   more than itself to the error, so that the moments of a peaked density, whose Hessian is badly
//   conditioned, are as good as FP64 sums (rounding down and adding the mean half unit back put half
//   a unit per point into them: up to 300 times the FP64 error in the Hessian's own metric).
// Written as plain C++ so that the host can check the arithmetic bit for bit.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define KITRT_FX __host__ __device__ __forceinline__
#else
#define KITRT_FX inline
struct int2 {
    int x, y;
};
#endif

namespace kitrt_fx {

constexpr int kFracBits = 42;             // fraction bits of the exponent s
constexpr float kFxMaxZ = 245.0f;         // sum_c |alpha_c| max|m_c| below this: |s| < 2^61.5
constexpr int kMaxShift = 32;             // largest power of two of a scaled row
constexpr int kGuard = 7;                 // y (2^62) >> 7 = 2^55

struct Limb {
    int h, l;
};

KITRT_FX long long wide(int a, int b) { return (long long)a * b; }
KITRT_FX uint32_t mulhi_u(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// y >> n for n >= 0, 0 when n >= 64; arithmetic version for signed sums.
KITRT_FX uint64_t shr(uint64_t y, int n)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(y), "r"(n));
    return r;
#else
    return n >= 64 ? 0 : y >> n;
#endif
}
KITRT_FX int imax(int a, int b) { return a > b ? a : b; }

// y / 2^n rounded to the nearest integer (halves up), n >= 1
KITRT_FX uint64_t shr_round(uint64_t y, int n) { return (shr(y, n - 1) + 1) >> 1; }
KITRT_FX long long sar(long long y, int n) { return y >> (n > 63 ? 63 : n); }

// v = h 2^B + l, |l| <= 2^(B - 1), for |v| < 2^(30 + B)
template <int B>
KITRT_FX Limb split(long long v)
{
    Limb r;
    r.h = (int)((v + (1LL << (B - 1))) >> B);
    r.l = (int)((uint32_t)v - (uint32_t)((uint64_t)(uint32_t)r.h << B));
    return r;
}

// Sum over k of A_k T_k (A_k: units of 2^-42, 31-bit limbs; T_k: units of 2^-54, 27-bit limbs).
struct DotAcc {
    long long hh = 0, hl = 1LL << 22, lh = 1LL << 26;
    KITRT_FX void add(Limb a, int2 t)
    {
        hh += wide(a.h, t.x);
        hl += wide(a.h, t.y);
        lh += wide(a.l, t.x);
    }
    KITRT_FX long long value() const { return (hh << 4) + (hl >> 23) + (lh >> 27); }
};

// Azimuthal sum of e T_k over up to 32 quads (e below 2^57 in magnitude, 27-bit limbs both), in
// units of e.
struct SumAcc {
    long long hh, m;
    KITRT_FX void clear() { hh = 0, m = 1LL << 26; }
    KITRT_FX void add(Limb e, int2 t)
    {
        hh += wide(e.h, t.x);
        m += wide(e.h, t.y);
        m += wide(e.l, t.x);
    }
    KITRT_FX long long value() const { return hh + (m >> 27); }
    KITRT_FX void scale_down(int n) { hh = sar(hh, n), m = sar(m, n); }
};

// One term B w P of a moment: B an azimuthal sum (below 2^62, split<32>), wP in units of 2^-57 (split<27>),
// in units of 2^sh of B (-20 < sh <= 2), rounded once.
KITRT_FX long long moment_term(Limb b, int2 wp, int sh)
{
    const long long t = (wide(b.h, wp.y) << 5) + wide(b.l, wp.x) + (wide(b.l, wp.y) >> 27);  // units 2^-30
    return (wide(b.h, wp.x) << (2 - sh)) + ((t + (1LL << (29 + sh))) >> (30 + sh));
}

// x 2^-sh as an integer in units of 2^-52, rounded (below 2048 in magnitude).
KITRT_FX long long fx_from_double(double x, int sh = 0)
{
    union {
        double d;
        uint64_t u;
    } b;
    b.d = x;
    const int ex = (int)((b.u >> 52) & 0x7ff) - 1023 - sh;
    const uint64_t mant = (b.u & 0xfffffffffffffULL) | (1ULL << 52);
    uint64_t v;
    if (ex >= 0) v = mant << (ex > 10 ? 10 : ex);
    else v = (shr(mant, -ex - 1) + 1) >> 1;
    return (b.u >> 63) ? -(long long)v : (long long)v;
}

// v 2^e as a double, rounded half away; 0 below the smallest normal double, infinite beyond the
// largest.
KITRT_FX double fx_to_double(long long v, int e)
{
    union {
        double d;
        uint64_t u;
    } b;
    const uint64_t sign = v < 0 ? 1ULL << 63 : 0;
    const uint64_t a = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)a);
#else
    const int lz = a ? __builtin_clzll(a) : 64;
#endif
    if (a == 0) return 0.0;
    // leading bit to bit 62, then 53 bits by adding half of the last kept bit
    const uint64_t n = lz >= 1 ? a << (lz - 1) : a >> 1;
    const uint64_t q = (n + (1ULL << 9)) >> 10;  // 2^52 <= q <= 2^53
    const int ex = e + (62 - (lz - 1)) + 1023;
    b.u = ex < 1 ? 0 : sign | (ex > 2046 ? 0x7ffULL << 52 : q + ((uint64_t)(ex - 1) << 52));
    return b.d;
}

// Sums of products alpha_c P_c of one exponent coefficient A_k: alpha_c in units of 2^-52 (split<32>),
// P_c in units of 2^-45 (split<27>).
struct CoefAcc {
    long long hh = 0, hl = 1LL << 22, lh = 1LL << 27, ll = 0;
    KITRT_FX void add(Limb a, int2 p)
    {
        hh += wide(a.h, p.x);
        hl += wide(a.h, p.y);
        lh += wide(a.l, p.x);
        ll += wide(a.l, p.y);
    }
    // in units of 2^-42
    KITRT_FX long long value() const { return (hh << 4) + (hl >> 23) + (lh >> 28) + (ll >> 55); }
};

// An exponential as (y, m): e = y 2^(m - 61).
struct Exp {
    uint64_t y;
    int m;
};

// 2^(s / 2048), s in units of 2^-42; tab[j] = 2^(j/2048) 2^61 rounded.
KITRT_FX Exp fx_exp(long long s, const uint64_t *tab)
{
    // L = ln2/2048 in units of 2^-56 with a quarter of the quartic coefficient; L^2/2, L^3/6 with
    // the rest of it (r^4 = 2 r^3 - 5/4 r^2 + r/4 - 1/128 + (at most 1/128) on [0, 1])
    constexpr uint64_t kC1 = 24387948313156ULL;
    constexpr uint32_t kC2 = 4127059915U, kC3 = 465681U;
    const int k = (int)(s >> 32) >> (kFracBits - 32);
    const uint32_t r = (uint32_t)(s >> (kFracBits - 32));            // fraction, 32 bits
    const uint32_t rl = (uint32_t)s & ((1u << (kFracBits - 32)) - 1);  // and 10 more
    const uint64_t T = tab[k & 2047];
    const uint32_t v = mulhi_u(r, mulhi_u(r, kC3) + kC2);
    const uint64_t g = kC1 + v;
    // p = r g in units of 2^-56 (below 2^44.5)
    uint64_t p = (uint64_t)r * (uint32_t)(g >> 32) + (((uint64_t)r * (uint32_t)g) >> 32);
    p += (rl * 5678u) >> 10;
    const uint32_t Th = (uint32_t)(T >> 32), Tl = (uint32_t)T;
    const uint32_t ph = (uint32_t)(p >> 32), pl = (uint32_t)p;
    Exp e;
    e.y = T + (((uint64_t)Th * ph) << 8) + (((uint64_t)Th * pl + (uint64_t)Tl * ph) >> 24);
    e.m = k >> 11;
    return e;
}

// The power of two by which a row is scaled down, from its bound sum_c |alpha_c| max|m_c|: 0 inside the
// range, the bound below 128 otherwise; -1 for one beyond 2^38 or not finite.
KITRT_FX int fx_row_shift(float bound)
{
    if (bound < kFxMaxZ) return 0;
    union {
        float f;
        uint32_t u;
    } b;
    b.f = bound;
    const int sh = (int)(b.u >> 23) - 127 - 6;
    return sh <= kMaxShift ? sh : -1;
}

// s 2^sh of a scaled row, 0 < sh <= kMaxShift: an s of 64 bits reaches as far as the doubles (-+ 709.78). As in
// kexp, exponents of -707 and below give no more than 2^-1024, which a double moment or ansatz has as
// 0. False, and the largest s, beyond the double range.
KITRT_FX bool fx_unscale(long long &s, int sh)
{
    const long long k = s >> (kFracBits - sh);
    const bool low = k <= -2088931, high = k > (1 << 21) - 1;  // -707 2048 / ln2; 2^21: 2^1024
    s = low ? INT64_MIN : high ? INT64_MAX : (long long)((uint64_t)s << sh);
    return !high;
}

// The same of an exponent in FP64 (NaN: false).
KITRT_FX bool fx_exponent_of(double z, long long &s)
{
    const bool ok = z < 709.78, live = ok && z > -707.0;
    s = live ? (long long)(z * (2954.639443740597 * 4398046511104.0)) : ok ? INT64_MIN : INT64_MAX;
    return ok;
}

// e as a float's bits, rounded half up; below the smallest normal float 0, beyond the range +inf.
KITRT_FX uint32_t fx_float_bits(Exp e)
{
    const uint32_t fb = (uint32_t)((e.y + (1ULL << 37)) >> 38);
    const uint32_t bits = fb + ((uint32_t)(e.m + 126) << 23);
    return e.m < -126 ? 0u : e.m > 127 ? 0x7f800000u : bits;
}

// e as a double, rounded half up (|m| far inside the double range).
KITRT_FX double fx_double(Exp e)
{
    union {
        double d;
        uint64_t u;
    } b;
    b.u = ((e.y + (1ULL << 8)) >> 9) + ((uint64_t)(e.m + 1022) << 52);
    return b.d;
}

// Exponent of the row scale from the zeroth moment the row is to reproduce: mean exponential
// u_0 / (4 pi m_0) = 0.282 u_0, and 2^4 above it; very low when u_0 says nothing (then the first
// pair decides).
KITRT_FX int fx_scale_of(double u0)
{
    union {
        double d;
        uint64_t u;
    } b;
    b.d = u0;
    const int ex = (int)(b.u >> 52);  // sign makes it large
    return ex == 0 || ex >= 0x7ff ? 100000 : ex - 1023 - 2 + 4 + kGuard;
}

// ---------------------------------------------------------------------------------------------
// One row's pass over the rule (sweep.cuh): exponent coefficients of a ring, exponents of a quad, azimuthal
// sums, moments.
// ---------------------------------------------------------------------------------------------
// Index of basis function (l, k), l + |k| even, in the order l ascending, then k ascending.
KITRT_FX constexpr int cindex(int l, int k) { return l * (l + 1) / 2 + (k + l) / 2; }

// Exponent coefficients of one ring: A0 (k = 0) and A[2(k-1)], A[2(k-1)+1] for cos(k phi),
// sin(k phi), from the trial alpha's limbs (at(c)).
template <int NN, typename At>
KITRT_FX void fx_coeffs(At &&at, const int2 *Pr, long long &A0, Limb (&A)[2 * NN])
{
#pragma unroll
    for (int k = -NN; k <= NN; ++k) {
        CoefAcc acc;
        const int ak = k < 0 ? -k : k;
#pragma unroll
        for (int l = ak; l <= NN; l += 2) acc.add(at(cindex(l, k)), Pr[cindex(l, k)]);
        const long long v = acc.value();
        if (k == 0) A0 = v;
        else A[2 * (ak - 1) + (k < 0)] = split<31>(v);
    }
}

// A row's azimuthal sums of the current ring, degree LB, and the exponent of their unit
// (units of 2^(Sx - 61)).
template <int LB>
struct FxSums {
    long long b0;
    SumAcc b[2 * LB];  // cos(k phi), sin(k phi) at 2(k-1), 2(k-1)+1
    int Sx;
    KITRT_FX void clear()
    {
        b0 = 0;
#pragma unroll
        for (int j = 0; j < 2 * LB; ++j) b[j].clear();
    }
};

// Moments of the finished ring: V_c += w_r P_c(mu_r) B_k(c), c over the degree-LB basis; the
// azimuthal sums are cleared for the next ring.
template <int LB, typename Acc>
KITRT_FX void fx_flush(const int2 *wPr, int sumshift, FxSums<LB> &B, Acc &&V)
{
#pragma unroll
    for (int k = -LB; k <= LB; ++k) {
        const int ak = k < 0 ? -k : k;
        const Limb v = split<32>(k == 0 ? B.b0 : B.b[k == 0 ? 0 : 2 * (ak - 1) + (k < 0)].value());
#pragma unroll
        for (int l = ak; l <= LB; l += 2) V(cindex(l, k)) += moment_term(v, wPr[cindex(l, k)], sumshift);
    }
    B.clear();
}

// The exponents of one quad's four points (t: its cosines, k = 1.., then from t + L2 its sines).
template <int NN>
KITRT_FX void fx_exponents(long long A0, const Limb (&A)[2 * NN], const int2 *t, int L2, bool axes, long long (&s)[4])
{
    long long ce = A0, co = 0, se = 0, so = 0;
    if (!axes) {
        DotAcc acc[4];  // C_e, C_o, S_e, S_o
#pragma unroll
        for (int k = 1; k <= NN; ++k) {
            acc[k & 1].add(A[2 * (k - 1)], t[k - 1]);
            acc[2 + (k & 1)].add(A[2 * (k - 1) + 1], t[L2 + k - 1]);
        }
        if (NN >= 2) ce += acc[0].value();
        co = acc[1].value();
        if (NN >= 2) se = acc[2].value();
        so = acc[3].value();
        const long long p = ce + co, m = ce - co, q = so + se, w = so - se;
        s[0] = p + q;
        s[1] = p - q;
        s[2] = m + w;
        s[3] = m - w;
    } else {
        // phi = 0, pi, pi/2, 3 pi/2: cos(k phi) and sin(k phi) are 0 and +-1
        long long ce2 = A0;
#pragma unroll
        for (int k = 1; k <= NN; ++k) {
            const long long a = ((long long)A[2 * (k - 1)].h << 31) + A[2 * (k - 1)].l;
            const long long b = ((long long)A[2 * (k - 1) + 1].h << 31) + A[2 * (k - 1) + 1].l;
            if (k & 1) {
                co += a;
                so += (k & 2) ? -b : b;
            } else {
                ce += a;
                ce2 += (k & 2) ? -a : a;
            }
        }
        s[0] = ce + co;
        s[1] = ce - co;
        s[2] = ce2 + so;
        s[3] = ce2 - so;
    }
}

// One quad's exponentials into the azimuthal sums. `first`: the row's first quad of this item
// (uniform), which lowers a scale that lies far above the row's exponentials. shift_moments(d)
// shifts the row's moments down by d when the scale rises.
template <int LB, typename Shift>
KITRT_FX void fx_accumulate(const Exp (&e)[4], const int2 *t, int L2, bool axes, bool first, FxSums<LB> &B,
                            Shift &&shift_moments)
{
    const int mm = imax(imax(e[0].m, e[1].m), imax(e[2].m, e[3].m));
    if (first && B.Sx - kGuard - mm > 22) B.Sx = mm + kGuard + 1;
    if (mm + kGuard > B.Sx) {
        const int d = mm + kGuard + 1 - B.Sx;
        B.Sx += d;
        B.b0 = sar(B.b0, d);
#pragma unroll
        for (int j = 0; j < 2 * LB; ++j) B.b[j].scale_down(d);
        shift_moments(d);
    }
    long long f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = (long long)shr_round(e[i].y, B.Sx - e[i].m);
    const long long p = f[0] + f[1], d = f[0] - f[1], p2 = f[2] + f[3], d2 = f[2] - f[3];
    const long long all = p + p2;
    B.b0 += all;
    if (!axes) {
        const Limb ce = split<27>(all), co = split<27>(p - p2);
        const Limb so = split<27>(d + d2), se = split<27>(d - d2);
#pragma unroll
        for (int k = 1; k <= LB; ++k) {
            B.b[2 * (k - 1)].add(k & 1 ? co : ce, t[k - 1]);
            B.b[2 * (k - 1) + 1].add(k & 1 ? so : se, t[L2 + k - 1]);
        }
    } else {
#pragma unroll
        for (int k = 1; k <= LB; ++k) {
            if (k & 1) {
                B.b[2 * (k - 1)].hh += d;
                B.b[2 * (k - 1) + 1].hh += (k & 2) ? -d2 : d2;
            } else {
                B.b[2 * (k - 1)].hh += (k & 2) ? p - p2 : all;
            }
        }
    }
}

}  // namespace kitrt_fx
