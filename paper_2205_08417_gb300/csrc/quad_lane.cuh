// A lane that owns one quad of azimuths of a cell (sweep.cuh) and walks the rings: shared by the FP64
// flux and the adjoint. 32 / J cells share a warp; lanes beyond them idle (coefficients 0).
#pragma once

#include "kitrt_internal.cuh"

namespace kitrt_quad {

// Tables of the quads (kitrt_mn_init), in double or float; the sqrt2 of T_k is in the ring tables.
template <typename F>
struct QuadTab {
    const F *ring;    // [R x n] w_r sin(theta_r) P_c(mu_r)
    const F *ringW;   // [R x n] w_r P_c(mu_r)
    const F *ringP;   // [R x n] P_c(mu_r)
    const F *ringS;   // [R] sin(theta_r)
    const F *az;      // [J x n] azimuthal factors of each quad, with the signs of the axes' quad
    const F *sc;      // [J x 2] sin, cos of phi_j
    const F *zrow;    // [Qp] zeros
    int R, P, J;
};

template <typename F>
inline QuadTab<F> quad_tab(const kitrt_mn *mn, const F *t)
{
    const size_t Rn = (size_t)mn->R * mn->n, Jn = (size_t)mn->J * mn->n;
    const F *s = t + 3 * Rn, *az = s + mn->R, *sc = az + Jn;
    return QuadTab<F>{t, t + Rn, t + 2 * Rn, s, az, sc, sc + 2 * mn->J, mn->R, mn->P, mn->J};
}
inline QuadTab<double> quad_tab64(const kitrt_mn *mn) { return quad_tab<double>(mn, mn->d_quad64); }
inline QuadTab<float> quad_tab32(const kitrt_mn *mn) { return quad_tab<float>(mn, mn->d_quad32); }

// The pairs A = (phi, pi + phi) and B = (-phi, pi - phi) of a lane's quad, or (0, pi) and
// (pi/2, 3 pi/2) for quad 0 (the axes; no B when the ring has an odd number of pairs): places in the
// ring's 2 P points, and sin, cos of each pair's first direction.
template <typename F>
struct QuadLane {
    bool live, axes, hasB;
    int ci, j;
    int oA1, oA2, oB1, oB2;
    F sA, cA, sB, cB;
    // lane: this thread's place among the `width` threads that share cells
    __device__ __forceinline__ QuadLane(const QuadTab<F> &X, int lane, int width = 32)
    {
        const int cpw = width / X.J, P = X.P;
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
        sB = axes ? F(1) : -sA;
        cB = axes ? F(0) : cA;
    }
};

// Two consecutive values as one access (the quad's pairs are 2-element aligned in every row whose
// length is even and whose base is).
__device__ __forceinline__ double2 pair_of(const double *p) { return *reinterpret_cast<const double2 *>(p); }
__device__ __forceinline__ float2 pair_of(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void pair_to(double *p, double a, double b) { *reinterpret_cast<double2 *>(p) = make_double2(a, b); }
__device__ __forceinline__ void pair_to(float *p, float a, float b) { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }

// The quad's four values A1, A2, B1, B2 of a row's ring: its two pairs of consecutive places hold
// (A1, B1) and (B2, A2), on the axes (A1, A2) and (B1, B2). (B1, B2 repeat the first pair when the
// quad has no B.)
template <typename F>
__device__ __forceinline__ void quad_load(const QuadLane<F> &Q, const F *p, F &a1, F &a2, F &b1, F &b2)
{
    const auto x = pair_of(p + Q.oA1);
    const auto y = pair_of(p + (Q.axes ? Q.oB1 : Q.oB2));
    a1 = x.x;
    a2 = Q.axes ? x.y : y.y;
    b1 = Q.axes ? y.x : x.y;
    b2 = Q.axes ? y.y : y.x;
}
template <typename F>
__device__ __forceinline__ void quad_store(const QuadLane<F> &Q, F *p, F a1, F a2, F b1, F b2)
{
    pair_to(p + Q.oA1, a1, Q.axes ? a2 : b1);
    if (Q.hasB) pair_to(p + (Q.axes ? Q.oB1 : Q.oB2), Q.axes ? b1 : b2, Q.axes ? b2 : a2);
}

// G_c += w_c v(c) for a quad whose pair sums and differences are ap = A1 + A2, am = A1 - A2, bp, bm: v(c)
// is the combination of the four values that cos(k phi) or sin(k phi) takes.
__device__ __forceinline__ double q_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float q_fma(float a, float b, float c) { return fmaf(a, b, c); }

template <int NN, typename F>
__device__ __forceinline__ void quad_project(bool axes, F ap, F am, F bp, F bm, const F *__restrict__ w,
                                             F (&G)[(NN + 1) * (NN + 2) / 2])
{
    const F all = ap + bp, even2 = ap - bp;
    const F v2 = axes ? even2 : all;  // cos, k = 2 mod 4
    const F oc = axes ? am : am + bm, os = axes ? bm : am - bm;
#pragma unroll
    for (int l = 0; l <= NN; ++l)
#pragma unroll
        for (int k = -l; k <= l; k += 2) {
            const int a = l * (l + 1) / 2 + (k + l) / 2;
            const F v = k >= 0 ? (k & 1 ? oc : k & 2 ? v2 : all) : (k & 1 ? os : even2);
            G[a] = q_fma(w[a], v, G[a]);
        }
}

// Values at the quad's four points (A1, A2, B1, B2) of sum_c P_c b_c, b_c = coefficient times the
// lane's azimuthal factor.
template <int NN, typename F>
__device__ __forceinline__ void quad_evaluate(bool axes, const F *__restrict__ P, const F (&b)[(NN + 1) * (NN + 2) / 2],
                                              F (&v)[4])
{
    F e0 = F(0), e2 = F(0), o = F(0), so = F(0), se = F(0);
#pragma unroll
    for (int l = 0; l <= NN; ++l)
#pragma unroll
        for (int k = -l; k <= l; k += 2) {
            const int a = l * (l + 1) / 2 + (k + l) / 2;
            F &t = k >= 0 ? (k & 1 ? o : k & 2 ? e2 : e0) : (k & 1 ? so : se);
            t = q_fma(P[a], b[a], t);
        }
    const F e = e0 + e2, p = e + o, m = e - o;
    if (axes) {
        const F x = e0 - e2;
        v[0] = p;
        v[1] = m;
        v[2] = x + so;
        v[3] = x - so;
    } else {
        const F q = so + se, w = so - se;
        v[0] = p + q;
        v[1] = m - w;
        v[2] = p - q;
        v[3] = m + w;
    }
}

}  // namespace kitrt_quad
