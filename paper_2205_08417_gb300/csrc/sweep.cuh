// Sum-factorised quadrature sums of the closure's dual on the folded product rule
// [Sec. 3.2, Eq. spherical-coordinatesProduct: Gauss-Legendre points in mu times equally spaced
// azimuths; Sec. 3.1: real spherical harmonics m_c = N_l^|k| P_l^|k|(mu) T_k(phi)].
//
// On a ring (one |mu|) every basis function is a Legendre factor times an azimuthal factor
// T_k(phi) (1, sqrt2 cos(k phi) or sqrt2 sin(|k| phi)), so
//   exponent   z(mu_r, phi) = alpha . m = sum_{k=-N..N} A_k(r) T_k(phi),
//              A_k(r) = sum_{c: k(c) = k} alpha_c P_c(mu_r)                 (once per ring),
//   moments    V_c = sum_r w_r P_c(mu_r) B_k(c)(r),  B_k(r) = sum_phi e(mu_r, phi) T_k(phi).
// The azimuths of a ring come in fours phi, -phi, pi - phi, pi + phi whose cosines and sines agree
// up to signs: with the even and odd parts of C = sum_{k>=0} A_k T_k and S = sum_{k<0} A_k T_k at phi,
//   z(+-phi) = (C_e + C_o) +- (S_o + S_e),   z(pi -+ phi) = (C_e - C_o) +- (S_o - S_e),
// and the azimuthal sums take the matching sums and differences of the four exponentials. A pass
// over a cell's Q' points then costs N/2 products per point for the exponent and L/2 for moments
// up to degree L, instead of n and nmom(L), plus n and nmom(L) per ring. The four azimuths 0, pi,
// pi/2, 3 pi/2 (only the first two when the number of pairs per ring is odd) need no products.
// The arithmetic is 64-bit fixed point (fixed.cuh): the FP64 pipe (16 cycles per warp instruction)
// bound the FP64 form of this pass. Measured on 99,458 cells, M_3, order 20 (400 folded points):
// tensor-core sweep 4.86 -> 1.53 ms for 350,160 cell evaluations, FP64-mode sweep 3.83 -> 0.86 ms
// for 219,742. Now bound by integer issue: about 25 32x32->64-bit products per point, each 4 cycles
// of the multiply pipe of a scheduler, and twice as many other instructions.
//
// Tables (built by kitrt_mn_init): ring r holds the folded points 2 P r .. 2 P (r + 1) - 1 in pairs
// (phi_j, -phi_j), phi_j = pi j / P, pair 0 being (0, pi); its quads are j = 0 (pair 0 and pair P/2)
// and j = 1 .. J - 1, J = (P + 1) / 2 rounded down (pairs j and P - j); quad qd = r J + j.
// fx_trig [J x 4N] limbs: cos(k phi_j), k = 1..2N, then sin(k phi_j).
// fx_ringA [R x n], fx_ringW [R x n2] limbs: P_c(mu_r) and w_r P_c(mu_r), both with the sqrt2 of
// T_k, the first times 2048/ln2, the second over 2^fx_wexp. fx_exp: 2^(j/2048) 2^61.
#pragma once

#include "fixed.cuh"
#include "kexp.cuh"
#include "kitrt_internal.cuh"

namespace kitrt_dev {

using kitrt_fx::cindex;
using kitrt_fx::Exp;
using kitrt_fx::fx_accumulate;
using kitrt_fx::fx_coeffs;
using kitrt_fx::fx_exponents;
using kitrt_fx::fx_flush;
using kitrt_fx::fx_row_shift;
using kitrt_fx::FxSums;
using kitrt_fx::Limb;

// The two pairs of points of quad j of a ring (the second is -1 in quad 0 of a ring with an odd
// number of pairs).
__device__ __forceinline__ int quad_pair0(int ring, int j, int P) { return ring * P + j; }
__device__ __forceinline__ int quad_pair1(int ring, int j, int P)
{
    return j ? ring * P + P - j : (P & 1) ? -1 : ring * P + P / 2;
}

// Where a row's trial point lies: a given alpha (phase NULL), or the Newton state's alpha + lam dir.
struct NewtonPoint {
    const double *alpha, *dir, *lam;
    const int32_t *phase;
};
__device__ __forceinline__ NewtonPoint point_of(const NewtonState &S, const double *given)
{
    return given ? NewtonPoint{given, given, nullptr, nullptr} : NewtonPoint{S.alpha, S.dir, S.lam, S.phase};
}

// The exponents s of a quad (points of pairs pa and pb) of a row outside the fixed-point range, in the units of
// the others: scaled back by 2^sh, or, for alpha of 1e11 or not finite (sh = -1), full FP64 sums against
// the basis. False when one is beyond the double range. The trial point (given, or that of the Newton
// state) is read again here, and the function is not inlined, so that the other rows carry none of
// it. Scaled rows take what the others take; FP64 exponents and exponentials (a thread per row, a few
// rows of a warp) held the FP64 pipe for 12 times the work of a warp per row.
template <int NN>
__device__ __noinline__ bool fx_outside(int sh, const double *__restrict__ Mt, int Qp, const NewtonPoint at, int cell,
                                        int pa, int pb, long long *s)
{
    constexpr int n = (NN + 1) * (NN + 2) / 2;
    bool ok = true;
    if (sh > 0) {
#pragma unroll
        for (int t = 0; t < 4; ++t) ok = kitrt_fx::fx_unscale(s[t], sh) && ok;
        return ok;
    }
    if (cell < 0) return true;  // a place without a cell
    const double *alpha = at.alpha + (size_t)cell * n, *dir = at.dir + (size_t)cell * n;
    const double lam = at.phase && at.phase[cell] == PH_NEWTON ? at.lam[cell] : 0.0;
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {
        const int q = 2 * (t < 2 ? pa : max(pb, 0)) + (t & 1);
        double z = 0.0;
#pragma unroll 1
        for (int c = 0; c < n; ++c) z = fma(lam != 0.0 ? fma(lam, dir[c], alpha[c]) : alpha[c], __ldg(Mt + (size_t)c * Qp + q), z);
        ok = kitrt_fx::fx_exponent_of(z, s[t]) && ok;
    }
    return ok;
}

// The same on registers: an array whose address goes to a function that is not inlined stays in local
// memory, and the other rows' exponents with it if it were the same one.
template <int NN>
__device__ __forceinline__ bool fx_outside_quad(int sh, const Tables &T, const NewtonPoint &at, int cell, int pa, int pb,
                                                long long (&s)[4])
{
    long long t[4] = {s[0], s[1], s[2], s[3]};
    const bool ok = fx_outside<NN>(sh, T.Mt, T.Qp, at, cell, pa, pb, t);
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] = t[i];
    return ok;
}

// Limbs of a row's trial alpha 2^-sh, components from, from + step, ...
__device__ __noinline__ static void fx_scale_limbs(const double *alpha, const double *dir, double lam, int from, int step,
                                                   int n, int sh, int2 *limbs, int pitch)
{
#pragma unroll 1
    for (int c = from; c < n; c += step) {
        const Limb w = kitrt_fx::split<32>(kitrt_fx::fx_from_double(lam != 0.0 ? fma(lam, dir[c], alpha[c]) : alpha[c], sh));
        limbs[c * pitch] = make_int2(w.h, w.l);
    }
}

// Exponent of the unit of a row's moments (for fx_to_double).
__device__ __forceinline__ int fx_unit(int Sx, const Tables &T) { return Sx - 61 + T.fx_sumshift + T.fx_wexp; }

// Conversions done in integer arithmetic, so that the narrow FP64 pipe does not execute them.
// Whether a double is finite (exponent field not all ones).
__device__ __forceinline__ bool finite_bits(double x)
{
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

// A finite double rounded to float: the exponent rebiased and the mantissa rounded half away from
// zero at bit 29 (a carry into the exponent is the correct result); magnitudes below the smallest
// normal float give a signed zero, magnitudes beyond the float range a signed infinity.
__device__ __forceinline__ float d2f_bits(double x)
{
    const long long b = __double_as_longlong(x);
    const long long mag = b & 0x7fffffffffffffffLL;
    const int sign = (int)((unsigned long long)b >> 32) & (int)0x80000000u;
    if ((int)(mag >> 52) < 1023 - 126) return __int_as_float(sign);
    long long f = ((mag + (1LL << 28)) >> 29) - ((long long)(1023 - 127) << 23);
    if (f >= (255LL << 23)) f = 255LL << 23;
    return __int_as_float((int)f | sign);
}

// A float widened to double exactly; subnormal floats give a signed zero, infinities and NaNs
// stay infinities and NaNs.
__device__ __forceinline__ double f2d_bits(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
    const unsigned mag = b & 0x7fffffffu;
    if (mag < 0x00800000u) return __longlong_as_double((long long)sign);
    if (mag >= 0x7f800000u)
        return __longlong_as_double((long long)(sign | 0x7ff0000000000000ULL |
                                                ((unsigned long long)(mag & 0x7fffffu) << 29)));
    return __longlong_as_double(
        (long long)(sign | (((unsigned long long)mag << 29) + ((unsigned long long)(1023 - 127) << 52))));
}

// Split of a sweep's work: tiles of 128 listed cells times parts of the quadrature (whole units of
// 4 quads in the FP64 sweeps, 8 in the tensor-core sweep; part j takes units
// [j nunits / parts, (j + 1) nunits / parts)). Part j of list slot i lands in column j * cnt + i of
// the accumulator, and the Newton kernels add the parts in order, so every cell's sums depend on the
// list's length only, not on its place (deterministic).
// The number of parts is the one with the shortest schedule on `grid` persistent CTAs, each item
// costing its units plus one for its trial point, its drain and its stores; at most
// 1 + target / tiles, which bounds the columns. Called by whole warps.
struct SweepSplit {
    int tiles, parts;
};
__device__ __forceinline__ SweepSplit sweep_split(int cnt, int grid, int target_items, int nunits)
{
    SweepSplit sp;
    sp.tiles = (cnt + 127) / 128;
    sp.parts = 1;
    if (target_items <= 0 || sp.tiles == 0) return sp;
    const int most = min(nunits, 1 + target_items / sp.tiles);
    unsigned best = 0xffffffffu;  // schedule length in the high bits, parts (at most 512) in the low 10
    for (int p = 1 + (threadIdx.x & 31); p <= most; p += 32) {
        const unsigned rounds = (unsigned)(sp.tiles * p + grid - 1) / grid;
        best = min(best, (rounds * ((nunits + p - 1) / p + 1)) << 10 | (unsigned)p);
    }
    sp.parts = (int)(__reduce_min_sync(0xffffffffu, best) & 1023u);
    return sp;
}

}  // namespace kitrt_dev
