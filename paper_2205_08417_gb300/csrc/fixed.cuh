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
//   with sum_c |alpha_c| max|m_c| >= kFxMaxZ take their exponentials from the FP64 kexp instead;
//   azimuthal factors cos(k phi), sin(k phi) in units of 2^-54, the weighted Legendre factors of
//   the moments in units of 2^-57 of a power of two, the exponent's in units of 2^-45;
//   exponential e = y 2^(m - 61), y in [2^61, 2^62]: T_j (1 + p) with the 2048-entry table and
//   p = exp(r ln2/2048) - 1 on r in [0, 1) by a cubic whose quartic term is folded in (error below
//   2^-57); |error| of y below 2^-51 relative;
//   sums in units of 2^(Sx - 61): e is shifted down by Sx - m >= 8, so that it stays below 2^54 and
//   32 quads fit; Sx belongs to the row and is raised (and the sums shifted) when a larger
//   exponential appears.
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
constexpr int kGuard = 8;                 // y (2^62) >> 8 = 2^54

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

// Azimuthal sum of e T_k over up to 32 quads (e below 2^56 in magnitude, 27-bit limbs both), in
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

// One term B w P of a moment: B an azimuthal sum (below 2^61, split<32>), wP in units of 2^-57 (split<27>),
// in units of 2^sh of B (0 <= sh <= 4).
KITRT_FX long long moment_term(Limb b, int2 wp, int sh)
{
    return ((wide(b.h, wp.x) << 2) >> sh) + ((wide(b.h, wp.y) + (1LL << (24 + sh))) >> (25 + sh)) +
           ((wide(b.l, wp.x) + (wide(b.l, wp.y) >> 27) + (1LL << (29 + sh))) >> (30 + sh));
}

// A double as an integer in units of 2^-52, rounded (|x| < 2048).
KITRT_FX long long fx_from_double(double x)
{
    union {
        double d;
        uint64_t u;
    } b;
    b.d = x;
    const int ex = (int)((b.u >> 52) & 0x7ff) - 1023;
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

// A non-negative double (kexp's result) as (y, m); 0 gives (0, very small m). Returns false for
// an infinity or NaN.
KITRT_FX bool fx_exp_from_double(double d, Exp &e)
{
    union {
        double d;
        uint64_t u;
    } b;
    b.d = d;
    const int ex = (int)(b.u >> 52);
    e.y = b.u ? ((b.u & 0xfffffffffffffULL) | (1ULL << 52)) << 9 : 0;
    e.m = b.u ? ex - 1023 : -100000;
    if (ex >= 0x7ff) {
        e.y = 1ULL << 61;
        e.m = 0;
        return false;
    }
    return true;
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

}  // namespace kitrt_fx
