// A lane that owns one quad of azimuths of a cell (sweep.cuh) and walks the rings: shared by the FP64
// flux and the adjoint. 32 / J cells share a warp; lanes beyond them idle (coefficients 0).
#pragma once

#include "kitrt_internal.cuh"

namespace kitrt_quad {

// Tables of the quads (kitrt_mn_init).
struct QuadTab {
    const double *ring;   // [R x n] w_r sin(theta_r) P_c(mu_r) (sqrt2 of T_k included)
    const double *ringP;  // [R x n] P_c(mu_r) (sqrt2 included)
    const double *az;     // [J x n] azimuthal factors of each quad, with the signs of the axes' quad
    const double *sc;     // [J x 2] sin, cos of phi_j
    const double *zrow;   // [Qp] zeros
    int R, P, J;
};

inline QuadTab quad_tab(const kitrt_mn *mn)
{
    return QuadTab{mn->d_flux_ring, mn->d_flux_ringP, mn->d_flux_az, mn->d_flux_sc, mn->d_zero64, mn->R, mn->P, mn->J};
}

// The pairs A = (phi, pi + phi) and B = (-phi, pi - phi) of a lane's quad, or (0, pi) and
// (pi/2, 3 pi/2) for quad 0 (the axes; no B when the ring has an odd number of pairs): places in the
// ring's 2 P points, and sin, cos of each pair's first direction.
struct QuadLane {
    bool live, axes, hasB;
    int ci, j;
    int oA1, oA2, oB1, oB2;
    double sA, cA, sB, cB;
    __device__ __forceinline__ QuadLane(const QuadTab &X, int lane)
    {
        const int cpw = 32 / X.J, P = X.P;
        live = lane < cpw * X.J;
        ci = live ? lane / X.J : cpw - 1;
        j = live ? lane - ci * X.J : 0;
        axes = j == 0;
        hasB = !axes || (P & 1) == 0;
        oA1 = axes ? 0 : 2 * j;
        oA2 = axes ? 1 : 2 * (P - j) + 1;
        oB1 = axes ? (hasB ? P : 0) : 2 * j + 1;
        oB2 = axes ? (hasB ? P + 1 : 0) : 2 * (P - j);
        sA = X.sc[2 * j];
        cA = X.sc[2 * j + 1];
        sB = axes ? 1.0 : -sA;
        cB = axes ? 0.0 : cA;
    }
};

// G_c += w_c v(c) for a quad whose pair sums and differences are ap = A1 + A2, am = A1 - A2, bp, bm: v(c)
// is the combination of the four values that cos(k phi) or sin(k phi) takes.
template <int NN>
__device__ __forceinline__ void quad_project(bool axes, double ap, double am, double bp, double bm,
                                             const double *__restrict__ w, double (&G)[(NN + 1) * (NN + 2) / 2])
{
    const double all = ap + bp, even2 = ap - bp;
    const double v2 = axes ? even2 : all;  // cos, k = 2 mod 4
    const double oc = axes ? am : am + bm, os = axes ? bm : am - bm;
#pragma unroll
    for (int l = 0; l <= NN; ++l)
#pragma unroll
        for (int k = -l; k <= l; k += 2) {
            const int a = l * (l + 1) / 2 + (k + l) / 2;
            const double v = k >= 0 ? (k & 1 ? oc : k & 2 ? v2 : all) : (k & 1 ? os : even2);
            G[a] = fma(w[a], v, G[a]);
        }
}

// Values at the quad's four points (A1, A2, B1, B2) of sum_c P_c b_c, b_c = coefficient times the
// lane's azimuthal factor.
template <int NN>
__device__ __forceinline__ void quad_evaluate(bool axes, const double *__restrict__ P,
                                              const double (&b)[(NN + 1) * (NN + 2) / 2], double (&v)[4])
{
    double e0 = 0.0, e2 = 0.0, o = 0.0, so = 0.0, se = 0.0;
#pragma unroll
    for (int l = 0; l <= NN; ++l)
#pragma unroll
        for (int k = -l; k <= l; k += 2) {
            const int a = l * (l + 1) / 2 + (k + l) / 2;
            double &t = k >= 0 ? (k & 1 ? o : k & 2 ? e2 : e0) : (k & 1 ? so : se);
            t = fma(P[a], b[a], t);
        }
    const double e = e0 + e2, p = e + o, m = e - o;
    if (axes) {
        const double x = e0 - e2;
        v[0] = p;
        v[1] = m;
        v[2] = x + so;
        v[3] = x - so;
    } else {
        const double q = so + se, w = so - se;
        v[0] = p + q;
        v[1] = m - w;
        v[2] = p - q;
        v[3] = m + w;
    }
}

}  // namespace kitrt_quad
