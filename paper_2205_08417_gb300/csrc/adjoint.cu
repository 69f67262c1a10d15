// Discrete adjoint of the FP64 M_N step, for the gradient of the absorbed energy in a target
// region with respect to per-block absorption and scattering coefficients.
//
// Step map [Sec. 4.2 explicit iteration, Sec. 4.4 kinetic flux, Sec. 3.1 isotropic scattering]:
//   u^{s+1}_i = u^s_i - dt/A_i F_i(psi(alpha(u^s))) + dt R_i(u^s_i),
//   R_i(u) = -sigma_a,i u - sigma_s,i (u - u_0 e_0) + q_i <m>.
// Objective: J = sum_{s<nsteps} dt sum_{i in target} A_i sigma_a,i <psi_i>, <psi_i> = u^s_i0 / m_0.
// Reverse sweep with lambda^{nsteps} = 0:
//   lambda^s_i = lambda^{s+1}_i + dt (-sigma_t,i lambda_i + sigma_s,i lambda_i0 e_0)
//              + H_i^-1 sum_q mu_iq psi_iq m_q + [i in target] dt A_i sigma_a,i / m_0 e_0,
// where d psi_iq / d u_i = psi_iq m_q^T H_i^-1 (implicit-function theorem on the closure, H the
// Hessian of the dual at the converged alpha) and mu_iq = d(sum_c lambda_c . u^{s+1}_c)/d psi_iq
// is the transposed upwind flux, gathered per cell from its own and its neighbours' lambda:
//   mu_iq = -dt w_q [ (L_iq/A_i) sum_f (Omega_q.n_if)(H_f + [Neumann boundary f](1 - H_f))
//                     - sum_{f interior} (L_jq/A_j) (Omega_q.n_if) H_f ],  L_cq = lambda_c . m_q,
// H_f = [Omega_q.n_if > 0]. Parameter gradients per block accumulate
//   dJ/dsigma_a += -dt lambda^{s+1}_i . u^s_i + [i in target] dt A_i u^s_i0 / m_0,
//   dJ/dsigma_s += -dt lambda^{s+1}_i . (u^s_i - u^s_i0 e_0).
// Memory: forward states are checkpointed every `ckpt_every` steps; each segment is recomputed
// forward (storing its alphas) before its reverse steps.
#include <math.h>
#include <string.h>

#include <vector>

#include "kexp.cuh"
#include "kitrt_internal.cuh"
#include "newton_common.cuh"
#include "quad_lane.cuh"

namespace {

using namespace kitrt_dev;
using namespace kitrt_quad;
constexpr int kWarps = 8;

__global__ void objective_kernel(const double *__restrict__ u, int n, const double *__restrict__ sa,
                                 const uint8_t *__restrict__ target, const double *__restrict__ area,
                                 double dt, double inv_m0, int C, double *__restrict__ J)
{
    double part = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x)
        if (target[i]) part += dt * area[i] * sa[i] * u[(size_t)i * n] * inv_m0;
    part = warp_sum(part);
    if ((threadIdx.x & 31) == 0 && part != 0.0) atomicAdd(J, part);
}

// The reverse step of one cell splits into four kernels, each in the layout that its work asks for:
//   moments and ansatz at the closed alpha   fixed-point sweep, a thread per cell (closure_fp64.cu)
//   L_cq = lambda_c . m_q / A_c              quads: the basis factorises into azimuth and ring
//   r_i = sum_q mu_iq psi_iq m_q             quads, as the FP64 flux (each face is outflow for exactly
//                                            one of a direction and its opposite)
//   H_i^-1 r_i, lambda, block gradients      8 lanes per cell, as the Newton step
// One kernel with a warp per cell did all of it in FP64 (70 FP64 instructions a point, 38 sums
// reduced over the warp, the factorisation with a row per lane): 59,168 cells, M_3, order 10:
// 3.05 -> 0.66 ms per reverse step.

template <int NN>
__global__ void __launch_bounds__(kWarps * 32)
lambda_dot_m_kernel(int Qp, QuadTab<double> X, const double *__restrict__ lam, const double *__restrict__ area,
                    double *__restrict__ Lq, int C)
{
    constexpr int n = Dims<NN>::n;
    extern __shared__ __align__(16) double lambda_smem[];  // [R x n] Legendre factors
    for (int e = threadIdx.x; e < X.R * n; e += blockDim.x) lambda_smem[e] = X.ringP[e];
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, cpw = 32 / X.J;
    const QuadLane<double> Q(X, lane);
    for (int base = (blockIdx.x * kWarps + wib) * cpw; base < C; base += gridDim.x * kWarps * cpw) {
        const int i = min(base + Q.ci, C - 1);
        const bool store = Q.live && base + Q.ci < C;
        const double inv = 1.0 / area[i];
        double b[n];
#pragma unroll
        for (int a = 0; a < n; ++a) b[a] = lam[(size_t)i * n + a] * inv * X.az[Q.j * n + a];
        double *row = Lq + (size_t)i * Qp;
#pragma unroll 1
        for (int r = 0; r < X.R; ++r, row += 2 * X.P) {
            double v[4];
            quad_evaluate<NN>(Q.axes, lambda_smem + r * n, b, v);
            if (store) {
                row[Q.oA1] = v[0];
                row[Q.oA2] = v[1];
                if (Q.hasB) {
                    row[Q.oB1] = v[2];
                    row[Q.oB2] = v[3];
                }
            }
        }
    }
}

template <int NN>
__global__ void __launch_bounds__(kWarps * 32, 2)
adjoint_flux_kernel(int Qp, QuadTab<double> X, const int4 *__restrict__ nbr, const double *__restrict__ nrm,
                    const double *__restrict__ psi, const double *__restrict__ Lq, double dt, int bc, int C,
                    double *__restrict__ rout)
{
    constexpr int n = Dims<NN>::n;
    extern __shared__ __align__(16) double adj_smem[];
    double *sR = adj_smem, *sT = sR + X.R * n, *sRed = sT + X.J * n;  // sRed [warp][n][32]
    for (int e = threadIdx.x; e < X.R * n; e += blockDim.x) sR[e] = X.ring[e];
    for (int e = threadIdx.x; e < X.J * n; e += blockDim.x) sT[e] = X.az[e];
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, J = X.J, cpw = 32 / J;
    double *red = sRed + wib * n * 32;
    const QuadLane<double> Q(X, lane);
    for (int base = (blockIdx.x * kWarps + wib) * cpw; base < C; base += gridDim.x * kWarps * cpw) {
        const int i = min(base + Q.ci, C - 1);
        const int4 nb = nbr[i];
        const int nbf[3] = {nb.x, nb.y, nb.z};
        const double *ps = psi + (size_t)i * Qp, *own = Lq + (size_t)i * Qp;
        const double *outA[3], *outB[3];
        double xA[3], xB[3];
        unsigned firstA = 0, firstB = 0;  // bit f: the face is outflow for the pair's first direction
        unsigned wall = 0;                // bit f: Neumann wall, whose ghost returns the cell's own psi
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const double nx = nrm[6 * (size_t)i + 2 * f], ny = nrm[6 * (size_t)i + 2 * f + 1];
            const double *row = nbf[f] >= 0 ? Lq + (size_t)nbf[f] * Qp : X.zrow;
            if (nbf[f] < 0 && bc == 0) wall |= 1u << f;
            const double dA = fma(nx, Q.sA, ny * Q.cA), dB = fma(nx, Q.sB, ny * Q.cB);
            const bool fA = dA > 0.0, fB = dB > 0.0;
            firstA |= (unsigned)fA << f;
            firstB |= (unsigned)fB << f;
            outA[f] = row + (fA ? Q.oA1 : Q.oA2);
            outB[f] = row + (fB ? Q.oB1 : Q.oB2);
            xA[f] = Q.live ? fabs(dA) : 0.0;
            xB[f] = Q.live && Q.hasB ? fabs(dB) : 0.0;
        }
        double G[n];
#pragma unroll
        for (int a = 0; a < n; ++a) G[a] = 0.0;
#pragma unroll 1
        for (int r = 0; r < X.R; ++r) {
            const int at = r * 2 * X.P;
            const double a1 = own[at + Q.oA1], a2 = own[at + Q.oA2], b1 = own[at + Q.oB1], b2 = own[at + Q.oB2];
            const double pa1 = ps[at + Q.oA1], pa2 = ps[at + Q.oA2], pb1 = ps[at + Q.oB1], pb2 = ps[at + Q.oB2];
            double ap = 0.0, am = 0.0, bp = 0.0, bm = 0.0;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const bool fA = (firstA >> f) & 1, fB = (firstB >> f) & 1;
                const double da = (fA ? a1 : a2) - outA[f][at], db = (fB ? b1 : b2) - outB[f][at];
                const double ca = xA[f] * (fA ? pa1 : pa2), cb = xB[f] * (fB ? pb1 : pb2);
                ap = fma(ca, da, ap);
                am = fma(fA ? ca : -ca, da, am);
                bp = fma(cb, db, bp);
                bm = fma(fB ? cb : -cb, db, bm);
            }
            if (wall) {
                // the wall's inflow: the other direction of each pair
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    if (!((wall >> f) & 1)) continue;
                    const bool fA = (firstA >> f) & 1, fB = (firstB >> f) & 1;
                    const double ta = xA[f] * (fA ? pa2 * a2 : pa1 * a1), tb = xB[f] * (fB ? pb2 * b2 : pb1 * b1);
                    ap -= ta;
                    am += fA ? ta : -ta;
                    bp -= tb;
                    bm += fB ? tb : -tb;
                }
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
            double v = 0.0;
            for (int t = 0; t < J; ++t) v += red[a * 32 + cc * J + t];
            rout[(size_t)ic * n + a] = -dt * v;
        }
    }
}

// lambda^s from lambda^{s+1}, and the block gradients: 8 lanes per cell, 32 cells per block and pass.
template <int NN>
__global__ void __launch_bounds__(kGroupBlock, 2)
adjoint_solve_kernel(Tables T, const double *__restrict__ V, int vs, const double *__restrict__ rin,
                     const double *__restrict__ u, const double *__restrict__ lam_next, const double *__restrict__ area,
                     const double *__restrict__ sa, const double *__restrict__ ss, const uint8_t *__restrict__ target,
                     const int32_t *__restrict__ block, double dt, int C, int nnz, double *__restrict__ lam,
                     double *__restrict__ gsa, double *__restrict__ gss, int32_t *__restrict__ fail)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, npairs = Dims<NN>::npairs, SL = (n + 7) / 8;
    extern __shared__ __align__(16) double solve_smem[];
    double *sV = solve_smem, *sH = sV + n2 * kGroupPitch, *coef = sH + kGroupCells * npairs;
    int32_t *gstart = reinterpret_cast<int32_t *>(coef + nnz);
    unsigned char *gidx = reinterpret_cast<unsigned char *>(gstart + npairs + 1);
    const int tid = threadIdx.x, lane = tid & 31, g = lane & 7, slot = tid >> 3;
    for (int t = tid; t < nnz; t += kGroupBlock) {
        gidx[t] = (unsigned char)T.gidx[t];
        coef[t] = T.gcoef[t];
    }
    for (int t = tid; t <= npairs; t += kGroupBlock) gstart[t] = T.gstart[t];
    for (int base = blockIdx.x * kGroupCells; base < C; base += gridDim.x * kGroupCells) {
        __syncthreads();
        for (int e = tid; e < n2 * kGroupCells; e += kGroupBlock) {
            const int c = e / kGroupCells, j = e % kGroupCells;
            sV[c * kGroupPitch + j] = V[(size_t)c * vs + min(base + j, C - 1)];
        }
        __syncthreads();
        const bool valid = base + slot < C;
        const int i = min(base + slot, C - 1);
        const size_t off = (size_t)i * n;
        double x[SL], li[SL], ua[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int c = g + 8 * s;
            x[s] = c < n ? rin[off + c] : 0.0;
            li[s] = c < n ? lam_next[off + c] : 0.0;
            ua[s] = c < n ? u[off + c] : 0.0;
        }
        const bool spd = group_factor_solve<NN, double>(coef, gidx, gstart, sV + slot, sH + slot * npairs, 0.0, n, g, x);
        const double l0 = __shfl_sync(kFull, li[0], 0, 8), u0 = __shfl_sync(kFull, ua[0], 0, 8);
        const double sai = sa[i], ssi = ss[i];
        const bool tgt = target[i] != 0;
        double lu = 0.0, lus = 0.0;
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int c = g + 8 * s;
            lu = fma(li[s], ua[s], lu);
            if (c > 0) lus = fma(li[s], ua[s], lus);
            if (valid && c < n) {
                double v = li[s] + dt * (-(sai + ssi) * li[s] + (c == 0 ? ssi * l0 : 0.0)) + (spd ? x[s] : 0.0);
                if (c == 0 && tgt) v += dt * area[i] * sai / T.m0;
                lam[off + c] = v;
            }
        }
        lu = group_sum(lu);
        lus = group_sum(lus);
        double da = -dt * lu + (tgt ? dt * area[i] * u0 / T.m0 : 0.0), ds = -dt * lus;
        if (!valid) da = ds = 0.0;
        if (g == 0 && valid && !spd) atomicAdd(fail, 1);
        // the warp's four cells mostly lie in one block: one atomic then
        const int blk = block[i];
        const bool one = __all_sync(kFull, blk == __shfl_sync(kFull, blk, 0));
        if (one) {
            da += __shfl_xor_sync(kFull, da, 8);
            ds += __shfl_xor_sync(kFull, ds, 8);
            da += __shfl_xor_sync(kFull, da, 16);
            ds += __shfl_xor_sync(kFull, ds, 16);
        }
        if (one ? lane == 0 : g == 0) {
            atomicAdd(&gsa[blk], da);
            atomicAdd(&gss[blk], ds);
        }
        __syncwarp();
    }
}

}  // namespace

// Device-side step used by the adjoint: closure (FP64, warm start), finish (alpha_out), flux.
// Declared in host.cu.
int kitrt_internal_step(kitrt_mn *mn, double *u, double *alpha, const double *sa, const double *ss,
                        const double *q, double dt, int first, cudaStream_t s);
int check_stability(kitrt_mn *mn, const double *sa, const double *ss, double dt, cudaStream_t s,
                    bool wait);

extern "C" int32_t kitrt_adjoint(kitrt_mn *mn, const double *u0, const double *alpha0,
                                 const double *sigma_a, const double *sigma_s, const double *q,
                                 const int32_t *block_of_cell, int32_t nblocks, const uint8_t *target,
                                 double dt, int32_t nsteps, int32_t ckpt_every, double *J,
                                 double *dJ_dsa, double *dJ_dss, void *stream)
{
    if (!mn || !u0 || !alpha0 || !sigma_a || !sigma_s || !q || !block_of_cell || !target || !J ||
        !dJ_dsa || !dJ_dss || nblocks < 1 || nsteps < 0 || ckpt_every < 1 || mn->p.mode != KITRT_FP64 ||
        mn->p.order != 1 || mn->p.reg_gamma != 0.0 || mn->d_invrho)
        return KITRT_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int C = mn->mesh->C, n = mn->n, Qp = mn->Qp;
    if (dt <= 0.0) dt = mn->p.cfl * mn->mesh->min_inradius;
    const size_t Cn = (size_t)C * n;
    const int nck = (nsteps + ckpt_every - 1) / ckpt_every;
    // the adjoint's buffers live in the solver's workspace: allocated by the first call that
    // needs them (or needs more than the last), kept for later calls, freed by kitrt_mn_destroy
    const size_t a256 = 255;
    const size_t sizes[] = {sizeof(double) * Cn * (nck > 0 ? nck : 1),  // ck_u
                            sizeof(double) * Cn * (nck > 0 ? nck : 1),  // ck_a
                            sizeof(double) * Cn * ckpt_every,           // seg_u
                            sizeof(double) * Cn * ckpt_every,           // seg_a
                            sizeof(double) * Cn, sizeof(double) * Cn,   // u, a
                            sizeof(double) * Cn, sizeof(double) * Cn,   // lam, lam2
                            sizeof(double) * (size_t)C * Qp,            // Lq
                            sizeof(double) * Cn,                        // r
                            sizeof(double) * (1 + 2 * (size_t)nblocks), // J, dJ_dsa, dJ_dss
                            sizeof(int32_t)};                           // fail
    constexpr int kBufs = sizeof(sizes) / sizeof(sizes[0]);
    size_t offs[kBufs], total = 0;
    for (int i = 0; i < kBufs; ++i) {
        offs[i] = total;
        total += (sizes[i] + a256) & ~a256;
    }
    if (mn->adj_bytes < total) {
        if (mn->d_adj) cudaFree(mn->d_adj);
        mn->d_adj = nullptr;
        mn->adj_bytes = 0;
        if (cudaMalloc(&mn->d_adj, total) != cudaSuccess) {
            mn->d_adj = nullptr;
            return KITRT_ENOMEM;
        }
        mn->adj_bytes = total;
    }
    unsigned char *base = (unsigned char *)mn->d_adj;
    double *ck_u = (double *)(base + offs[0]);
    double *ck_a = (double *)(base + offs[1]);
    double *seg_u = (double *)(base + offs[2]);
    double *seg_a = (double *)(base + offs[3]);
    double *u = (double *)(base + offs[4]);
    double *a = (double *)(base + offs[5]);
    double *lam = (double *)(base + offs[6]);
    double *lam2 = (double *)(base + offs[7]);
    double *Lq = (double *)(base + offs[8]);
    double *r = (double *)(base + offs[9]);
    double *dJ = (double *)(base + offs[10]);  // J, then dJ/dsigma_a, then dJ/dsigma_s
    double *dJ_sa = dJ + 1, *dJ_ss = dJ + 1 + nblocks;
    int32_t *fail = (int32_t *)(base + offs[11]);
    auto cleanup = [](int rc) { return rc; };
    int rc0 = check_stability(mn, sigma_a, sigma_s, dt, s, true);
    if (rc0) return rc0;
    const Tables T = mn->tables();
    const kitrt_mesh *m = mn->mesh;
    const double inv_m0 = 1.0 / T.m0;
    const int tb = (C + 255) / 256 < mn->nsm * 8 ? (C + 255) / 256 : mn->nsm * 8;
    const QuadTab<double> X = quad_tab64(mn);
    const int per_block = kWarps * (32 / mn->J), qb = std::min((C + per_block - 1) / per_block, mn->nsm * 2);
    const int lb = std::min((C + per_block - 1) / per_block, mn->nsm * 8);
    const int sb = std::min((C + kGroupCells - 1) / kGroupCells, mn->nsm * 2);
    const size_t smem_l = sizeof(double) * mn->R * n, smem_f = sizeof(double) * n * ((size_t)mn->R + mn->J + kWarps * 32);
    const size_t smem_s = group_smem_bytes(mn->n2, mn->npairs, mn->gaunt_nnz, false);
#define CK(x)                                          \
    do {                                               \
        if ((x) != cudaSuccess) return cleanup(KITRT_ECUDA); \
    } while (0)
    CK(cudaMemsetAsync(dJ, 0, sizeof(double) * (1 + 2 * (size_t)nblocks), s));
    CK(cudaMemsetAsync(fail, 0, sizeof(int32_t), s));
    CK(cudaMemcpyAsync(u, u0, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
    CK(cudaMemcpyAsync(a, alpha0, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
    // forward sweep: objective and checkpoints (state and warm start at each segment start)
    for (int st = 0; st < nsteps; ++st) {
        if (st % ckpt_every == 0) {
            CK(cudaMemcpyAsync(ck_u + Cn * (st / ckpt_every), u, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
            CK(cudaMemcpyAsync(ck_a + Cn * (st / ckpt_every), a, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
        }
        {
            LaunchScope ls(mn, PK_ADJOINT, s, C);
            objective_kernel<<<tb, 256, 0, s>>>(u, n, sigma_a, target, m->d_area, dt, inv_m0, C, dJ);
        }
        const int rc = kitrt_internal_step(mn, u, a, sigma_a, sigma_s, q, dt, st == 0, s);
        if (rc) return cleanup(rc);
    }
    // reverse sweep, segment by segment
    CK(cudaMemsetAsync(lam, 0, sizeof(double) * Cn, s));
    for (int seg = nck - 1; seg >= 0; --seg) {
        const int s0 = seg * ckpt_every, s1 = (s0 + ckpt_every < nsteps) ? s0 + ckpt_every : nsteps;
        CK(cudaMemcpyAsync(u, ck_u + Cn * seg, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(a, ck_a + Cn * seg, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
        for (int st = s0; st < s1; ++st) {
            CK(cudaMemcpyAsync(seg_u + Cn * (st - s0), u, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
            const int rc = kitrt_internal_step(mn, u, a, sigma_a, sigma_s, q, dt, st == s0, s);
            if (rc) return cleanup(rc);
            // a holds the converged alpha of u^st after the step
            CK(cudaMemcpyAsync(seg_a + Cn * (st - s0), a, sizeof(double) * Cn, cudaMemcpyDeviceToDevice, s));
        }
        for (int st = s1 - 1; st >= s0; --st) {
            const double *us = seg_u + Cn * (st - s0), *as = seg_a + Cn * (st - s0);
            const int rc = launch_adjoint_closure(mn, T, C, us, as, mn->d_Vacc, mn->vs, mn->d_psi, s);
            if (rc) return cleanup(rc);
            LaunchScope ls(mn, PK_ADJOINT, s, C);
            mn->launch_count += 2;  // three kernels in this scope
#define ADJ_CASE(NNv)                                                                                          \
    case NNv:                                                                                                  \
        if (ensure_dyn_smem(adjoint_flux_kernel<NNv>, smem_f) || ensure_dyn_smem(adjoint_solve_kernel<NNv>, smem_s)) \
            return cleanup(KITRT_ECUDA);                                                                       \
        lambda_dot_m_kernel<NNv><<<lb, kWarps * 32, smem_l, s>>>(Qp, X, lam, m->d_area, Lq, C);                \
        adjoint_flux_kernel<NNv><<<qb, kWarps * 32, smem_f, s>>>(Qp, X, m->d_nbr, m->d_nrm, mn->d_psi, Lq, dt, \
                                                                 mn->p.bc, C, r);                              \
        adjoint_solve_kernel<NNv><<<sb, kGroupBlock, smem_s, s>>>(T, mn->d_Vacc, mn->vs, r, us, lam, m->d_area, \
                                                                  sigma_a, sigma_s, target, block_of_cell, dt, \
                                                                  C, mn->gaunt_nnz, lam2, dJ_sa, dJ_ss, fail); \
        break;
            switch (mn->N) {
                ADJ_CASE(1)
                ADJ_CASE(2)
                ADJ_CASE(3)
                ADJ_CASE(4)
                ADJ_CASE(5)
            default: return cleanup(KITRT_EINVAL);
            }
#undef ADJ_CASE
            CK(cudaGetLastError());
            double *t = lam;
            lam = lam2;
            lam2 = t;
        }
    }
    int32_t nf = 0;
    CK(cudaMemcpyAsync(&nf, fail, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(J, dJ, sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(dJ_dsa, dJ_sa, sizeof(double) * nblocks, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(dJ_dss, dJ_ss, sizeof(double) * nblocks, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
#undef CK
    return cleanup(nf ? KITRT_ECHOL : KITRT_OK);
}
