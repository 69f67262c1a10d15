// Kinetic upwind flux of the closed ansatz and the explicit first-order update
// [Sec. 4.4 kinetic numerical flux; Sec. 4.2 explicit iteration; Sec. 3.1 isotropic scattering].
//
// Cell-centric gather (lanes over the folded quadrature points of a cell). The upwind
// flux sum_f sum_q w_q m_q (Omega_q.n_f) psi_up is evaluated in its fluctuation form
//     F_i = sum_f sum_{q: Omega_q.n_f < 0} w_q m_q (Omega_q.n_f) (psi_up,f,q - psi_iq),
// which equals it exactly in exact arithmetic because the scaled normals of a closed cell sum to
// zero (sum_f n_f = 0), so psi_iq sum_f Omega_q.n_f vanishes: outflow directions drop out, the
// upwind value is the neighbour's psi (the ghost: psi_iq for Neumann, 0 for vacuum), and a
// uniform state gives exactly zero flux at any working precision. F is projected on the basis,
// warp-reduced, and u <- u - dt/A F + dt R(u) is applied in place (the flux reads psi only).
// psi rows are contiguous per cell, so each face gather is a coalesced row segment.
#include <string.h>

#include "flux_group.cuh"
#include "kitrt_internal.cuh"
#include "quad_lane.cuh"

namespace {

using namespace kitrt_flux;
using namespace kitrt_quad;
constexpr int kWarps = 8;

// FP64 flux (FP64 mode). The FP64 pipe is the bound (a warp-wide FP64 instruction holds it for 16
// cycles), so the kernel is laid out for few of them: 32 per quad of points instead of 22 per point.
//  - A lane owns one quad of azimuths (sweep.cuh: phi, -phi, pi - phi, pi + phi) of its cell and walks
//    the rings; 32 / J cells share a warp. Omega.n_f = sin(theta_r) d_f(phi), so the face coefficients
//    d_f are formed once per lane and sin(theta_r) w_r goes into the ring table.
//  - d_f changes sign between a direction and its opposite, so each face is inflow for exactly one
//    of phi and pi + phi (and of -phi and pi - phi): three face terms per such pair, read at the point
//    that takes them.
//  - The basis factorises: with the sums and differences of the quad's four values the projection
//    takes one FMA per moment, ring and lane, and the azimuthal factor one product per moment at
//    the end.
// Measured on 99,458 cells, M_3, order 20: 1.72 -> 0.73 ms a step, of which 0.59 ms is the FP64 pipe
// at 16 cycles for each of the 347 warp instructions of three cells.
// RHO: the transformed CSD equation's density (Sec. 2, Eq. BoltzmannCSDTrafo): the transported
// value is psi / rho, so each row is scaled by its cell's 1/rho (invrho) before differencing.
template <int NN, bool RHO>
__global__ void __launch_bounds__(kWarps * 32, 2)
flux64_kernel(Tables T, QuadTab<double> X, const int4 *__restrict__ nbr, const double *__restrict__ nrm,
              const double *__restrict__ area, const double *__restrict__ psi,
              const double *__restrict__ invrho, double *__restrict__ u,
              const double *__restrict__ sa, const double *__restrict__ ss,
              const double *__restrict__ qs, double dt, int bc, int C)
{
    constexpr int n = (NN + 1) * (NN + 2) / 2;
    extern __shared__ __align__(16) double flux_smem[];
    double *sR = flux_smem, *sT = sR + X.R * n, *sRed = sT + X.J * n;  // sRed [warp][n][32]
    for (int e = threadIdx.x; e < X.R * n; e += blockDim.x) sR[e] = X.ring[e];
    for (int e = threadIdx.x; e < X.J * n; e += blockDim.x) sT[e] = X.az[e];
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int J = X.J, P = X.P, cpw = 32 / J;  // cells per warp
    const int Qp = T.Qp;
    double *red = sRed + wib * n * 32;
    const QuadLane<double> Q(X, lane);
    for (int base = (blockIdx.x * kWarps + wib) * cpw; base < C; base += gridDim.x * kWarps * cpw) {
        const int i = min(base + Q.ci, C - 1);
        const int4 nb = nbr[i];
        const int nbf[3] = {nb.x, nb.y, nb.z};
        const double *own = psi + (size_t)i * Qp;
        const double ri = RHO ? invrho[i] : 1.0;
        const double *upA[3], *upB[3];
        double cA[3], cB3[3], g[3];
        unsigned firstA = 0, firstB = 0;  // bit f: the face is inflow for the pair's first direction
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const double nx = nrm[6 * (size_t)i + 2 * f], ny = nrm[6 * (size_t)i + 2 * f + 1];
            // upwind row: the neighbour's, or on the boundary the cell's own as the ghost (Neumann:
            // fluctuation exactly 0) or zeros (vacuum: fluctuation -psi_i)
            const double *row = nbf[f] >= 0 ? psi + (size_t)nbf[f] * Qp : bc == 0 ? own : X.zrow;
            g[f] = RHO && nbf[f] >= 0 ? invrho[nbf[f]] : ri;
            const double dA = fma(nx, Q.sA, ny * Q.cA), dB = fma(nx, Q.sB, ny * Q.cB);
            const bool fA = __double2hiint(dA) < 0, fB = __double2hiint(dB) < 0;
            firstA |= (unsigned)fA << f;
            firstB |= (unsigned)fB << f;
            upA[f] = row + (fA ? Q.oA1 : Q.oA2);
            upB[f] = row + (fB ? Q.oB1 : Q.oB2);
            cA[f] = Q.live ? -fabs(dA) : 0.0;
            cB3[f] = Q.live && Q.hasB ? -fabs(dB) : 0.0;
            // a Neumann ghost's scaled difference would leave a rounding residue: the face drops out
            if (RHO && nbf[f] < 0 && bc == 0) cA[f] = cB3[f] = 0.0;
        }
        double G[n];
#pragma unroll
        for (int a = 0; a < n; ++a) G[a] = 0.0;
#pragma unroll 1
        for (int r = 0; r < X.R; ++r) {
            const int at = r * 2 * P;
            double a1 = own[at + Q.oA1], a2 = own[at + Q.oA2], b1 = own[at + Q.oB1], b2 = own[at + Q.oB2];
            double wA[3], wB[3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                wA[f] = upA[f][at];
                wB[f] = upB[f][at];
            }
            if (RHO) {
                a1 *= ri;
                a2 *= ri;
                b1 *= ri;
                b2 *= ri;
            }
            // sums and differences over each pair of the upwind fluctuations
            double ap = 0.0, am = 0.0, bp = 0.0, bm = 0.0;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const bool fA = (firstA >> f) & 1, fB = (firstB >> f) & 1;
                const double oa = fA ? a1 : a2, ob = fB ? b1 : b2;
                const double da = RHO ? fma(g[f], wA[f], -oa) : wA[f] - oa;
                const double db = RHO ? fma(g[f], wB[f], -ob) : wB[f] - ob;
                ap = f ? fma(cA[f], da, ap) : cA[f] * da;
                am = f ? fma(fA ? cA[f] : -cA[f], da, am) : (fA ? ap : -ap);
                bp = f ? fma(cB3[f], db, bp) : cB3[f] * db;
                bm = f ? fma(fB ? cB3[f] : -cB3[f], db, bm) : (fB ? bp : -bp);
            }
            quad_project<NN>(Q.axes, ap, am, bp, bm, sR + r * n, G);
        }
        __syncwarp();
#pragma unroll
        for (int a = 0; a < n; ++a) red[a * 32 + lane] = G[a] * sT[Q.j * n + a];
        __syncwarp();
        for (int e = lane; e < cpw * n; e += 32) {
            const int cc = e / n, a = e - cc * n, ic = base + cc;
            if (ic >= C) continue;
            double Fa = 0.0;
            for (int t = 0; t < J; ++t) Fa += red[a * 32 + cc * J + t];
            const double u0 = a == 0 ? u[(size_t)ic * n] : 0.0;
            const double ua = u[(size_t)ic * n + a];
            const double R = -sa[ic] * ua - ss[ic] * (ua - u0) + qs[ic] * T.mbar[a];
            u[(size_t)ic * n + a] = ua - dt / area[ic] * Fa + dt * R;
        }
    }
}

// FP32 flux of the mixed modes. FP64 instructions are rare on this GPU (2 per clock per SM), so
// none is spent on warp-uniform values: normals and inverse areas come from the mesh's FP32
// copies, the per-cell coefficients are converted by different lanes at once, and the update
// increment dt (-F/A + R(u)) is formed in FP32; only u += increment is FP64 (lanes over the
// (cell, moment) elements of a warp's cells).
//
// Layout of the work: a group of kGroup = 8 lanes takes two neighbouring cells, 8 cells per warp. Each
// lane reads 16-byte pieces (4 consecutive points) of each cell's row and of its three upwind rows,
// and the matching pieces of the tables once for both cells (the warp's groups read them at the
// same addresses: one request serves them). Q' padded to a multiple of 32 gives every lane the same
// number of pieces. Each lane sums its points in plain FP32; the 8 lane sums of a cell are reduced
// with a compensated (two-sum) reduce-scatter.
// Upwind fluctuation sum of one point: s = sum_f min(Omega.n_f, 0) (psi_up,f - psi_i), or with a
// density (RHO) sum_f min(Omega.n_f, 0) (psi_up,f / rho_up,f - psi_i / rho_i) (r: the 1/rho).
template <bool RHO>
__device__ __forceinline__ float point_fluct(float wx, float wy, const float (&nx)[3],
                                             const float (&ny)[3], float ri, const float (&r)[3],
                                             float pi, float u0, float u1, float u2)
{
    if (RHO) {
        const float tp = ri * pi;
        float s = fminf(fmaf(wx, nx[0], wy * ny[0]), 0.0f) * fmaf(r[0], u0, -tp);
        s = fmaf(fminf(fmaf(wx, nx[1], wy * ny[1]), 0.0f), fmaf(r[1], u1, -tp), s);
        return fmaf(fminf(fmaf(wx, nx[2], wy * ny[2]), 0.0f), fmaf(r[2], u2, -tp), s);
    }
    float s = fminf(fmaf(wx, nx[0], wy * ny[0]), 0.0f) * (u0 - pi);
    s = fmaf(fminf(fmaf(wx, nx[1], wy * ny[1]), 0.0f), u1 - pi, s);
    return fmaf(fminf(fmaf(wx, nx[2], wy * ny[2]), 0.0f), u2 - pi, s);
}

// L1 is the bound: with one cell per group 12 of the 16 pieces that a lane reads per 4 points are
// tables (n basis rows and w Omega). M_3, 99,458 cells 0.127 -> 0.126 ms (there latency
// counts as much: half the warps), M_5, 996,872 cells 4.8 -> 3.1 ms. Every sum keeps the order it had. (A
// factorised form by quads, as the FP64 flux, took 0.082 ms, but its other order of FP32 sums moved u
// by up to 1e-8 on coarse meshes.)
constexpr int kPair = 2;                                 // cells per group
constexpr int kCells32 = kPair * kCellsPerWarp;          // cells per warp
template <int NN, bool RHO>
__global__ void __launch_bounds__(kWarps * 32, 2)
flux_update32_kernel(Tables T, const int4 *__restrict__ nbr, const float *__restrict__ nrm32,
                     const float *__restrict__ inva32, const float *__restrict__ psi,
                     const float *__restrict__ zrow, const float *__restrict__ invrho32,
                     double *__restrict__ u,
                     const double *__restrict__ sa, const double *__restrict__ ss,
                     const double *__restrict__ qs, float dt, int bc, int C)
{
    constexpr int n = (NN + 1) * (NN + 2) / 2;
    constexpr int K = GroupRS<n>::K;
    __shared__ float sF[kWarps][kCells32 * n];
    __shared__ float sK[kWarps][kCells32][4];  // per cell: sigma_a, sigma_s, q, 1/A (FP32)
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int grp = lane >> kGroupLog, gl = lane & (kGroup - 1);
    const int Qp = T.Qp, nq4 = Qp / 4;
    const float4 *__restrict__ wx4 = reinterpret_cast<const float4 *>(T.wox32);
    const float4 *__restrict__ wy4 = reinterpret_cast<const float4 *>(T.woy32);
    const float4 *__restrict__ M4 = reinterpret_cast<const float4 *>(T.Mt32);
    for (int base = (blockIdx.x * kWarps + wib) * kCells32; base < C; base += gridDim.x * kWarps * kCells32) {
        const int nb_cells = C - base < kCells32 ? C - base : kCells32;
        if (lane < 4 * nb_cells) {
            const int ci = lane >> 2, which = lane & 3, i = base + ci;
            const double v = which == 0 ? sa[i] : which == 1 ? ss[i] : qs[i];
            sK[wib][ci][which] = which == 3 ? inva32[i] : (float)v;
        }
        float nx[kPair][3], ny[kPair][3], r[kPair][3], ri[kPair];
        const float4 *own[kPair], *up[kPair][3];
#pragma unroll
        for (int t = 0; t < kPair; ++t) {
            // a place without a cell repeats the warp's last one; its sums are not stored
            const int i = base + (kPair * grp + t < nb_cells ? kPair * grp + t : nb_cells - 1);
            const int4 nb = nbr[i];
            const int nbf[3] = {nb.x, nb.y, nb.z};
            own[t] = reinterpret_cast<const float4 *>(psi + (size_t)i * Qp);
            ri[t] = RHO ? invrho32[i] : 1.0f;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                nx[t][f] = nrm32[6 * (size_t)i + 2 * f];
                ny[t][f] = nrm32[6 * (size_t)i + 2 * f + 1];
                r[t][f] = RHO && nbf[f] >= 0 ? invrho32[nbf[f]] : ri[t];
                if (RHO && nbf[f] < 0 && bc == 0) nx[t][f] = ny[t][f] = 0.0f;  // Neumann ghost drops out
                // upwind row: the neighbour's; on the boundary the cell's own (Neumann ghost:
                // fluctuation 0) or the zero row (vacuum ghost: fluctuation -psi_i)
                up[t][f] = nbf[f] >= 0 ? reinterpret_cast<const float4 *>(psi + (size_t)nbf[f] * Qp)
                           : bc == 0   ? own[t]
                                       : reinterpret_cast<const float4 *>(zrow);
            }
        }
        float F[kPair][n];
#pragma unroll
        for (int t = 0; t < kPair; ++t)
#pragma unroll
            for (int a = 0; a < n; ++a) F[t][a] = 0.0f;
#pragma unroll 1
        for (int j = gl; j < nq4; j += kGroup) {
            float4 po[kPair], pu[kPair][3];
#pragma unroll
            for (int t = 0; t < kPair; ++t) {
                po[t] = __ldg(own[t] + j);
#pragma unroll
                for (int f = 0; f < 3; ++f) pu[t][f] = __ldg(up[t][f] + j);
            }
            const float4 wx = __ldg(wx4 + j), wy = __ldg(wy4 + j);
            float s[kPair][4];
#pragma unroll
            for (int t = 0; t < kPair; ++t) {
                s[t][0] = point_fluct<RHO>(wx.x, wy.x, nx[t], ny[t], ri[t], r[t], po[t].x, pu[t][0].x, pu[t][1].x, pu[t][2].x);
                s[t][1] = point_fluct<RHO>(wx.y, wy.y, nx[t], ny[t], ri[t], r[t], po[t].y, pu[t][0].y, pu[t][1].y, pu[t][2].y);
                s[t][2] = point_fluct<RHO>(wx.z, wy.z, nx[t], ny[t], ri[t], r[t], po[t].z, pu[t][0].z, pu[t][1].z, pu[t][2].z);
                s[t][3] = point_fluct<RHO>(wx.w, wy.w, nx[t], ny[t], ri[t], r[t], po[t].w, pu[t][0].w, pu[t][1].w, pu[t][2].w);
            }
#pragma unroll
            for (int a = 0; a < n; ++a) {
                const float4 m = __ldg(M4 + (size_t)a * nq4 + j);
#pragma unroll
                for (int t = 0; t < kPair; ++t)
                    F[t][a] = fmaf(m.w, s[t][3], fmaf(m.z, s[t][2], fmaf(m.y, s[t][1], fmaf(m.x, s[t][0], F[t][a]))));
            }
        }
#pragma unroll
        for (int t = 0; t < kPair; ++t) {
            float rs[K], re[K];
            int slot0;
            const bool uniq = group_reduce_scatter<n>(F[t], gl, rs, re, slot0);
            const int ci = kPair * grp + t;
            if (ci < nb_cells && uniq) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (slot0 + k < n) sF[wib][ci * n + slot0 + k] = rs[k] + re[k];
            }
        }
        __syncwarp();
        for (int idx = lane; idx < nb_cells * n; idx += 32) {
            const int ci = idx / n, a = idx - ci * n, ic = base + ci;
            const double ua = u[(size_t)ic * n + a];
            const float *k = sK[wib][ci];
            // R = -sigma_a u - sigma_s (u - u_0 e_0) + q <m>: the scattering term of moment 0
            // cancels exactly
            const float sig = a == 0 ? k[0] : k[0] + k[1];
            const float R = fmaf(-sig, (float)ua, k[2] * T.mbar32[a]);
            const float inc = dt * fmaf(-k[3], sF[wib][idx], R);
            u[(size_t)ic * n + a] = ua + (double)inc;
        }
        __syncwarp();
    }
}

}  // namespace

int launch_flux_update(kitrt_mn *mn, const Tables &T, int C, const double *psi,
                       const float *psi32, double *u, const double *sa, const double *ss,
                       const double *q, double dt, int bc, cudaStream_t s)
{
    const kitrt_mesh *m = mn->mesh;
    const QuadTab<double> X = quad_tab64(mn);
    const int per_block = kWarps * (32 / mn->J), need = (C + per_block - 1) / per_block;
    const int grid = need < mn->nsm * 2 ? (need > 0 ? need : 1) : mn->nsm * 2;
    const size_t smem64 = sizeof(double) * mn->n * ((size_t)mn->R + mn->J + kWarps * 32);
    const int need32 = (C + kWarps * kCells32 - 1) / (kWarps * kCells32);
    const int most32 = mn->nsm * 2, grid32 = need32 < most32 ? (need32 > 0 ? need32 : 1) : most32;  // persistent
    if (!psi && (T.Qp % 32 != 0 || !mn->d_zero32)) return KITRT_EINVAL;
    const bool rho = mn->d_invrho != nullptr;
    LaunchScope ls(mn, PK_FLUX, s, C);
#define FLUX_LAUNCH(NN, R)                                                                     \
    if (psi) {                                                                                 \
        if (ensure_dyn_smem(flux64_kernel<NN, R>, smem64)) return KITRT_ECUDA;                 \
        flux64_kernel<NN, R><<<grid, kWarps * 32, smem64, s>>>(                                \
            T, X, m->d_nbr, m->d_nrm, m->d_area, psi, mn->d_invrho, u, sa, ss, q, dt, bc, C);  \
    } else {                                                                                   \
        flux_update32_kernel<NN, R><<<grid32, kWarps * 32, 0, s>>>(                            \
            T, m->d_nbr, m->d_nrm32, m->d_inva32, psi32, mn->d_zero32, mn->d_invrho32, u, sa,  \
            ss, q, (float)dt, bc, C);                                                          \
    }
#define FLUX_CASE(NN)                                                                          \
    case NN:                                                                                   \
        if (rho) {                                                                             \
            FLUX_LAUNCH(NN, true)                                                              \
        } else {                                                                               \
            FLUX_LAUNCH(NN, false)                                                             \
        }                                                                                      \
        break;
    switch (mn->N) {
        FLUX_CASE(1)
        FLUX_CASE(2)
        FLUX_CASE(3)
        FLUX_CASE(4)
        FLUX_CASE(5)
    default: return KITRT_EINVAL;
    }
#undef FLUX_LAUNCH
#undef FLUX_CASE
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// Stability of the explicit step. The first-order kinetic update of the ansatz at quadrature
// point q keeps psi_iq (1 - dt/A_i sum_f (Omega_q.n_f)^+ - dt sigma_t,i) of the cell's own value;
// for a triangle sum_f (Omega.n_f)^+ = 1/2 sum_f |Omega.n_f| <= P_i / 2, so
//     dt (P_i / (2 A_i) + sigma_a,i + sigma_s,i) <= 1
// in every cell keeps every updated ordinate a non-negative combination of non-negative values
// (scattering and source only add), and the updated moments realizable. This is the cell-wise
// form of dt sigma_t,max <= 1 - CFL with CFL = dt / min_i (2 A_i / P_i), which implies it. With a
// density (transported value psi / rho) the outflow rate of cell i is P_i / (2 A_i rho_i).
namespace {

__global__ void stability_kernel(const double *__restrict__ hpa, const double *__restrict__ invrho,
                                 const double *__restrict__ sa, const double *__restrict__ ss,
                                 double dt, int C, unsigned long long *__restrict__ out)
{
    double worst = 0.0;
    unsigned bad = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x) {
        const double a = sa[i], b = ss[i];
        // with a density the transport speed of cell i is 1 / rho_i
        const double h = invrho ? hpa[i] * invrho[i] : hpa[i];
        if (!(a >= 0.0) || !(b >= 0.0) || !isfinite(a) || !isfinite(b)) ++bad;
        else worst = fmax(worst, dt * (h + a + b));
    }
    // non-negative doubles order like their bit patterns
    unsigned long long wb = __double_as_longlong(worst);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, wb, o);
        wb = x > wb ? x : wb;
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&out[0], wb);
        if (bad) atomicAdd(&out[1], (unsigned long long)bad);
    }
}

}  // namespace

int check_stability(kitrt_mn *mn, const double *sa, const double *ss, double dt, cudaStream_t s,
                    bool wait)
{
    const int C = mn->mesh->C;
    if (!(dt > 0.0) || !isfinite(dt)) return KITRT_EINVAL;
    if (cudaMemsetAsync(mn->d_check, 0, 2 * sizeof(unsigned long long), s) != cudaSuccess)
        return KITRT_ECUDA;
    int blocks = (C + 255) / 256;
    if (blocks > mn->nsm * 4) blocks = mn->nsm * 4;
    {
        LaunchScope ls(mn, PK_OTHER, s, C);
        stability_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(mn->mesh->d_hpa, mn->d_invrho, sa,
                                                                  ss, dt, C, mn->d_check);
    }
    if (cudaGetLastError() != cudaSuccess) return KITRT_ECUDA;
    if (cudaMemcpyAsync(mn->h_check, mn->d_check, 2 * sizeof(unsigned long long),
                        cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return KITRT_ECUDA;
    if (!wait) return KITRT_OK;
    if (cudaStreamSynchronize(s) != cudaSuccess) return KITRT_ECUDA;
    return stability_verdict(mn);
}

// Reads the test's result (the stream must have passed the copy in check_stability).
int stability_verdict(const kitrt_mn *mn)
{
    if (mn->h_check[1] != 0) return KITRT_EINVAL;
    double worst;
    memcpy(&worst, &mn->h_check[0], sizeof(double));
    // a relative slack of 1e-12 keeps dt = 1 / max(...) itself admissible after rounding
    return worst <= 1.0 + 1e-12 ? KITRT_OK : KITRT_EINVAL;
}
