// S_N step of the nodal (discrete-ordinates) system [Sec. 2, Eq. SNEqns2], explicit first-order
// finite volumes [Sec. 4.2] with the upwind flux applied to every ordinate [Sec. 4.4]:
//   psi'_iq = psi_iq - dt/A_i sum_f (Omega_q . n_if) psi_up - dt sigma_t,i psi_iq
//             + dt (O Sigma_i M psi_i)_q + dt q_i,
// on the solver's folded quadrature (the +-mu ordinates of the 2D problem are equal, so one
// folded point of weight 2w carries both). The scattering is the P_N form of Eq. SNEqns2
// truncated at the solver's degree N: the n moments M psi_i = sum_q w_q m(Omega_q) psi_iq are
// scaled by sigma_s,i g_l(a) (g_0 = 1) and mapped back by O = m(Omega_q); sigma_t = sigma_a +
// sigma_s. Isotropic scattering keeps the zeroth moment only.
//
// The flux is evaluated in fluctuation form, sum over faces with Omega.n < 0 of
// (Omega.n)(psi_up - psi_i), which equals the upwind form because the scaled normals of a closed
// cell sum to zero; a uniform state then sees exactly zero transport.
//
// Layout (quad_lane.cuh): a lane owns one quad of azimuths (phi, -phi, pi - phi, pi + phi) of its cell
// and walks the rings, once for the moments and once for the update (whose own values are then in
// L1); 32 / J cells share a warp. Omega.n = sin(theta_r) d_f(phi): the face coefficients are formed
// once per lane, each face is inflow for exactly one direction of an opposite pair, and the
// moments and the scattering factorise into azimuth and ring. That leaves, per ordinate, about 8
// (isotropic) or 17 (10 moments) FP64 instructions instead of 20 or 40, in FP32 2 paired and 6
// scalar loads per quad instead of 4 rows and the tables. Measured against the former kernel (tiles staged by
// bulk copies, a warp per cell), per step: FP32, isotropic, 99,458 cells, 400 ordinates 0.157 ->
// 0.100 ms (3.3 TB/s of the 326 MB that have to move); FP64, 10 moments, 20,000 cells, 240 ordinates
// 0.456 -> 0.231 ms.
#include <math.h>
#include <stdint.h>

#include "kitrt_internal.cuh"
#include "quad_lane.cuh"

namespace {

using namespace kitrt_quad;

constexpr int kWarps = 8;

// Per-basis-function scattering coefficient g_l(a), a < n, in the ordinates' precision.
template <typename P>
struct SnScat {
    P ga[KITRT_MAX_NMOM];
};

// Per-cell coefficients of the step in the ordinates' precision, formed once per call so that
// the step itself has no FP64 work in FP32 mode: scaled normals of the three faces, dt / A_i,
// 1 - dt sigma_t,i, dt q_i and sigma_s,i (12 slots, the last two unused).
constexpr int kCellSlots = 12;
template <typename P>
__global__ void sn_cell_prep_kernel(const double *__restrict__ nrm, const double *__restrict__ area,
                                    const double *__restrict__ sa, const double *__restrict__ ss,
                                    const double *__restrict__ qs, double dt, P *__restrict__ cell, int C)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x) {
        P *c = cell + (size_t)i * kCellSlots;
#pragma unroll
        for (int k = 0; k < 6; ++k) c[k] = (P)nrm[6 * (size_t)i + k];
        c[6] = (P)(dt / area[i]);
        c[7] = (P)(1.0 - dt * (sa[i] + ss[i]));
        c[8] = (P)(dt * qs[i]);
        c[9] = (P)ss[i];
        c[10] = P(0);
        c[11] = P(0);
    }
}

// Dynamic shared memory: the ring tables (w P, and P when anisotropic; sin theta), the azimuthal
// factors (anisotropic), and per warp [nm x 32] sums and [32 / J x nm] scattered moments; with a block per
// group of cells [nm x 256] sums, then [cells x nm] and [split x cells x nm], at most 256 nm / J each.
inline size_t sn_smem(size_t size, int R, int J, int n, bool iso)
{
    const int nm = iso ? 1 : n;
    return size * ((size_t)R * nm * (iso ? 1 : 2) + R + (iso ? 0 : (size_t)J * n) + (size_t)nm * std::max(kWarps * 64, 256 + 512 / J));
}

// How the step's work is laid out. A warp with 32 / J cells of its own walks their rings, twice, without a
// block barrier: best where there are cells for every warp. On a small mesh that is one chain of R
// rings in a few blocks, and for J > 10 it leaves up to 15 lanes idle: there a block takes
// 256 / (split J) cells together and its threads divide the rings into `split` parts. Eight warps of
// an SM keep its FP64 pipe busy, so that the time goes with the blocks of the fullest SM, each of its
// rings and two more for coefficients and sums (three with the block's barriers); the layout with the
// least of that is taken. In FP32 a warp with its own cells is taken throughout (its sums keep their order).
// FP64, 10 moments, ms a step, warp -> block: 338 cells, order 20 0.061 -> 0.020; 722 cells, order 15
// 0.053 -> 0.022; 3,362 cells, order 34 0.36 -> 0.18; 10,082 cells, order 22 0.31 -> 0.26, order 34
// 0.82 -> 0.47. 20,000 cells, order 15 (J = 8) keep the warp: 0.231.
struct SnLayout {
    int split;   // 0: a warp per group of cells
    int blocks;
};
inline SnLayout sn_layout(int C, int R, int J, int nsm, bool fp64)
{
    const int most = nsm * (fp64 ? 2 : 3), per_block = kWarps * (32 / J), need = (C + per_block - 1) / per_block;
    SnLayout best{0, std::min(need, most)};
    if (!fp64) return best;
    long cost = (long)((need + nsm - 1) / nsm) * (R + 2);
    for (int split = 1; split <= 8 && split <= R && 32 * kWarps / split >= J; split *= 2) {
        const int cells = 32 * kWarps / split / J, blocks = (C + cells - 1) / cells;
        const long c = (long)((blocks + nsm - 1) / nsm) * ((R + split - 1) / split + 3);
        if (c < cost) {
            cost = c;
            best = SnLayout{split, std::min(blocks, most)};
        }
    }
    return best;
}

template <typename P, int NN, bool ISO, bool BLOCK>
__global__ void __launch_bounds__(kWarps * 32, sizeof(P) == 4 ? 3 : 2)
sn_quad_kernel(QuadTab<P> X, int Qf, const int4 *__restrict__ nbr, const P *__restrict__ cellc,
               const P *__restrict__ psi, P *__restrict__ out, SnScat<P> sc, P dts, int bc, int C, int split)
{
    constexpr int n = (NN + 1) * (NN + 2) / 2, nm = ISO ? 1 : n;
    extern __shared__ __align__(16) unsigned char sn_smem_raw[];
    // threads that share cells and their number of cells; the first ring of this thread and their distance
    const int J = X.J, width = BLOCK ? 32 * kWarps / split : 32, cpw = width / J;
    const int part = BLOCK ? threadIdx.x / width : 0, step = BLOCK ? split : 1;
    P *sW = reinterpret_cast<P *>(sn_smem_raw);  // [R][nm] w P
    P *sS = sW + X.R * nm;                       // [R] sin theta
    P *sP = sS + X.R;                            // [R][n] P (anisotropic)
    P *sT = sP + (ISO ? 0 : X.R * n);            // [J][n] azimuthal factors (anisotropic)
    P *sRed = sT + (ISO ? 0 : J * n);            // [warp][2][nm][32]
    for (int e = threadIdx.x; e < X.R * nm; e += blockDim.x) sW[e] = X.ringW[ISO ? e * n : e];
    for (int e = threadIdx.x; e < X.R; e += blockDim.x) sS[e] = X.ringS[e];
    if (!ISO) {
        for (int e = threadIdx.x; e < X.R * n; e += blockDim.x) sP[e] = X.ringP[e];
        for (int e = threadIdx.x; e < J * n; e += blockDim.x) sT[e] = X.az[e];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int pitch = BLOCK ? 32 * kWarps : 32, at0 = BLOCK ? threadIdx.x : lane;  // of the sums
    P *red = BLOCK ? sRed : sRed + wib * nm * 64, *mom = red + nm * pitch, *sums = mom + cpw * nm;
    const QuadLane<P> Q(X, BLOCK ? threadIdx.x - part * width : lane, width);
    const int groups = BLOCK ? gridDim.x : gridDim.x * kWarps;
    for (int base = (BLOCK ? blockIdx.x : blockIdx.x * kWarps + wib) * cpw; base < C; base += groups * cpw) {
        const int i = min(base + Q.ci, C - 1);
        const bool store = Q.live && base + Q.ci < C;
        const P *own = psi + (size_t)i * Qf;
        const P *cf = cellc + (size_t)i * kCellSlots;
        const int4 nb = nbr[i];
        const int nbf[3] = {nb.x, nb.y, nb.z};
        // face coefficients -|d|; the face is inflow for the pair's first direction (bit f set) or its
        // second, and the upwind value is read at that direction's place
        const P *upA[3], *upB[3];
        P xA[3], xB[3];
        unsigned firstA = 0, firstB = 0;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const P nx = cf[2 * f], ny = cf[2 * f + 1];
            // neighbour, or on the boundary the cell's own row (Neumann: fluctuation 0) or zeros (vacuum)
            const P *row = nbf[f] >= 0 ? psi + (size_t)nbf[f] * Qf : bc == 0 ? own : X.zrow;
            const P dA = q_fma(nx, Q.sA, ny * Q.cA), dB = q_fma(nx, Q.sB, ny * Q.cB);
            const bool fA = dA < P(0), fB = dB < P(0);
            firstA |= (unsigned)fA << f;
            firstB |= (unsigned)fB << f;
            upA[f] = row + (fA ? Q.oA1 : Q.oA2);
            upB[f] = row + (fB ? Q.oB1 : Q.oB2);
            xA[f] = fA ? dA : -dA;
            xB[f] = fB ? dB : -dB;
        }
        // moments
        P G[nm];
#pragma unroll
        for (int a = 0; a < nm; ++a) G[a] = P(0);
#pragma unroll 2
        for (int r = part; r < X.R; r += step) {
            const P *p = own + r * 2 * X.P;
            P a1, a2, b1, b2;
            quad_load(Q, p, a1, a2, b1, b2);
            if (!Q.hasB) b1 = b2 = P(0);
            if constexpr (ISO)
                G[0] = q_fma(sW[r], (a1 + a2) + (b1 + b2), G[0]);
            else
                quad_project<NN, P>(Q.axes, a1 + a2, a1 - a2, b1 + b2, b1 - b2, sW + r * n, G);
        }
        const P dtA = cf[6], keep = cf[7], src = cf[8], sig_s = cf[9];
        auto barrier = [] {
            if constexpr (BLOCK) __syncthreads();
            else __syncwarp();
        };
        // (a block's sums of the former cells were read before its last two barriers)
        if constexpr (!BLOCK) __syncwarp();
#pragma unroll
        for (int a = 0; a < nm; ++a) red[a * pitch + at0] = ISO ? G[a] : G[a] * sT[ISO ? 0 : Q.j * n + a];
        barrier();
        if constexpr (BLOCK) {
            // the J sums of each part, then the parts
            for (int e = threadIdx.x; e < split * cpw * nm; e += 32 * kWarps) {
                const int sp = e / (cpw * nm), cc = (e - sp * cpw * nm) / nm, a = e % nm;
                P v = P(0);
                for (int t = 0; t < J; ++t) v += red[a * pitch + sp * width + cc * J + t];
                sums[e] = v;
            }
            __syncthreads();
            for (int e = threadIdx.x; e < cpw * nm; e += 32 * kWarps) {
                P v = P(0);
                for (int sp = 0; sp < split; ++sp) v += sums[sp * cpw * nm + e];
                mom[e] = ISO ? v : sc.ga[e % nm] * v;
            }
            __syncthreads();
        } else if constexpr (!ISO) {
            for (int e = lane; e < cpw * n; e += 32) {
                const int cc = e / n, a = e - cc * n;
                P v = P(0);
                for (int t = 0; t < J; ++t) v += red[a * 32 + cc * J + t];
                mom[cc * n + a] = sc.ga[a] * v;
            }
            __syncwarp();
        }
        P b[nm], iso = P(0);  // scattered moments times the lane's azimuthal factors
        if constexpr (ISO) {
            if constexpr (BLOCK) iso = mom[Q.ci];
            else
                for (int t = 0; t < J; ++t) iso += red[Q.ci * J + t];
            // dt (O Sigma M psi + q): sigma_s m_0 (sum_q w_q m_0 psi_q), the ring table holds w m_0
            iso = q_fma(dts * sig_s * X.ringP[0], iso, src);
        } else {
#pragma unroll
            for (int a = 0; a < nm; ++a) b[a] = mom[Q.ci * n + a] * (dts * sig_s) * sT[Q.j * n + a];
        }
        // update
        P *o = out + (size_t)i * Qf;
#pragma unroll(sizeof(P) == 4 ? 2 : 1)
        for (int r = part; r < X.R; r += step) {
            const int at = r * 2 * X.P;
            P a1, a2, b1, b2;
            quad_load(Q, own + at, a1, a2, b1, b2);
            P fa1 = P(0), fa2 = P(0), fb1 = P(0), fb2 = P(0);
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const bool fA = (firstA >> f) & 1, fB = (firstB >> f) & 1;
                const P da = upA[f][at] - (fA ? a1 : a2), db = upB[f][at] - (fB ? b1 : b2);
                fa1 = q_fma(fA ? xA[f] : P(0), da, fa1);
                fa2 = q_fma(fA ? P(0) : xA[f], da, fa2);
                fb1 = q_fma(fB ? xB[f] : P(0), db, fb1);
                fb2 = q_fma(fB ? P(0) : xB[f], db, fb2);
            }
            P s[4];
            if constexpr (ISO) {
                s[0] = s[1] = s[2] = s[3] = iso;
            } else {
                quad_evaluate<NN, P>(Q.axes, sP + r * n, b, s);
#pragma unroll
                for (int t = 0; t < 4; ++t) s[t] += src;
            }
            const P c = -dtA * sS[r];
            if (store)
                quad_store(Q, o + at, q_fma(keep, a1, q_fma(c, fa1, s[0])), q_fma(keep, a2, q_fma(c, fa2, s[1])),
                           q_fma(keep, b1, q_fma(c, fb1, s[2])), q_fma(keep, b2, q_fma(c, fb2, s[3])));
        }
    }
}

template <typename P, int NN, bool ISO, bool BLOCK>
int launch_sn_as(kitrt_mn *mn, const QuadTab<P> &X, const P *psi, P *out, const P *cellc, const SnScat<P> &sc, double dt,
                 const SnLayout &lay, cudaStream_t s)
{
    const kitrt_mesh *m = mn->mesh;
    const size_t smem = sn_smem(sizeof(P), mn->R, mn->J, mn->n, ISO);
    if (ensure_dyn_smem(sn_quad_kernel<P, NN, ISO, BLOCK>, smem)) return KITRT_ECUDA;
    LaunchScope ls(mn, PK_SN, s, m->C);
    sn_quad_kernel<P, NN, ISO, BLOCK><<<lay.blocks, kWarps * 32, smem, s>>>(X, mn->Qf, m->d_nbr, cellc, psi, out, sc,
                                                                            (P)dt, mn->p.bc, m->C, lay.split);
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

template <typename P, int NN, bool ISO>
int launch_sn(kitrt_mn *mn, const QuadTab<P> &X, const P *psi, P *out, const P *cellc, const SnScat<P> &sc,
              double dt, cudaStream_t s)
{
    const SnLayout lay = sn_layout(mn->mesh->C, mn->R, mn->J, mn->nsm, sizeof(P) == 8);
    if constexpr (sizeof(P) == 8)
        if (lay.split) return launch_sn_as<P, NN, ISO, true>(mn, X, psi, out, cellc, sc, dt, lay, s);
    return launch_sn_as<P, NN, ISO, false>(mn, X, psi, out, cellc, sc, dt, lay, s);
}

template <typename P, bool ISO>
int dispatch_sn(kitrt_mn *mn, const QuadTab<P> &X, const P *psi, P *out, const P *cellc,
                const SnScat<P> &sc, double dt, cudaStream_t s)
{
    switch (mn->N) {
    case 1: return launch_sn<P, 1, ISO>(mn, X, psi, out, cellc, sc, dt, s);
    case 2: return launch_sn<P, 2, ISO>(mn, X, psi, out, cellc, sc, dt, s);
    case 3: return launch_sn<P, 3, ISO>(mn, X, psi, out, cellc, sc, dt, s);
    case 4: return launch_sn<P, 4, ISO>(mn, X, psi, out, cellc, sc, dt, s);
    case 5: return launch_sn<P, 5, ISO>(mn, X, psi, out, cellc, sc, dt, s);
    default: return KITRT_EINVAL;
    }
}

template <typename P>
int run_sn(kitrt_mn *mn, const QuadTab<P> &X, P *psi, P *work, P *cellc, const double *sa, const double *ss,
           const double *q, const SnScat<P> &sc, bool iso, double dt, int nsteps, cudaStream_t s)
{
    const kitrt_mesh *m = mn->mesh;
    {
        int blocks = (m->C + 255) / 256;
        if (blocks > mn->nsm * 8) blocks = mn->nsm * 8;
        LaunchScope ls(mn, PK_OTHER, s, m->C);
        sn_cell_prep_kernel<P><<<blocks > 0 ? blocks : 1, 256, 0, s>>>(m->d_nrm, m->d_area, sa, ss, q, dt,
                                                                        cellc, m->C);
        if (cudaGetLastError() != cudaSuccess) return KITRT_ECUDA;
    }
    P *a = psi, *b = work;
    for (int it = 0; it < nsteps; ++it) {
        const int rc = iso ? dispatch_sn<P, true>(mn, X, a, b, cellc, sc, dt, s)
                           : dispatch_sn<P, false>(mn, X, a, b, cellc, sc, dt, s);
        if (rc) return rc;
        P *t = a;
        a = b;
        b = t;
    }
    // an odd number of steps leaves the result in the scratch buffer
    if (a != psi &&
        cudaMemcpyAsync(psi, a, sizeof(P) * (size_t)mn->mesh->C * mn->Qf, cudaMemcpyDeviceToDevice,
                        s) != cudaSuccess)
        return KITRT_ECUDA;
    return KITRT_OK;
}

}  // namespace

extern "C" {

int32_t kitrt_sn_step(kitrt_mn *mn, void *psi, void *work, int32_t fp32, const double *sigma_a,
                      const double *sigma_s, const double *q, const double *g, double dt,
                      int32_t nsteps, void *stream)
{
    if (!mn || !psi || !work || !sigma_a || !sigma_s || !q || nsteps < 0 || mn->d_invrho)
        return KITRT_EINVAL;
    if (((uintptr_t)psi | (uintptr_t)work) & 15) return KITRT_EINVAL;
    const size_t bytes = (fp32 ? 4 : 8) * (size_t)mn->mesh->C * mn->Qf;
    const uintptr_t pa = (uintptr_t)psi, pb = (uintptr_t)work;
    if (pa < pb + bytes && pb < pa + bytes) return KITRT_EINVAL;  // the buffers overlap
    double ga[KITRT_MAX_NMOM] = {};
    bool iso = true;
    {
        // degree of each basis function, in the basis order (l ascending, then k)
        int a = 0;
        for (int l = 0; l <= mn->N; ++l)
            for (int k = -l; k <= l; ++k) {
                if ((l + (k < 0 ? -k : k)) % 2) continue;
                const double gl = g ? g[l] : (l == 0 ? 1.0 : 0.0);
                if (l == 0 && gl != 1.0) return KITRT_EINVAL;
                if (!isfinite(gl)) return KITRT_EINVAL;
                if (l > 0 && gl != 0.0) iso = false;
                ga[a++] = gl;
            }
    }
    if (nsteps == 0) return KITRT_OK;
    cudaStream_t s = (cudaStream_t)stream;
    if (dt <= 0.0) dt = mn->p.cfl * mn->mesh->min_inradius;
    // The per-cell coefficients lie in the solver's workspace, which a call on another stream would
    // overwrite: every call waits on its stream (not on the host) for the end of the one before. A
    // captured call cannot wait for work outside its graph, and a replay overlaps anything: its
    // coefficients lie in memory of the graph's own.
    cudaStreamCaptureStatus capture;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) return KITRT_ECUDA;
    const bool captured = capture != cudaStreamCaptureStatusNone;
    void *cellc = mn->d_sn_cell;
    if (captured) {
        if (cudaMallocAsync(&cellc, (fp32 ? 4 : 8) * (size_t)mn->mesh->C * kCellSlots, s) != cudaSuccess)
            return KITRT_ENOMEM;
    }
    unsigned long long id = 0;  // of the stream, unlike its handle never used again
    if (!captured) {
        if (cudaStreamGetId(s, &id) != cudaSuccess) return KITRT_ECUDA;
        if (mn->sn_pending && id != mn->sn_stream && cudaStreamWaitEvent(s, mn->sn_done, 0) != cudaSuccess)
            return KITRT_ECUDA;
    }
    int rc;
    if (fp32) {
        SnScat<float> sc{};
        for (int a = 0; a < KITRT_MAX_NMOM; ++a) sc.ga[a] = (float)ga[a];
        rc = run_sn<float>(mn, quad_tab32(mn), (float *)psi, (float *)work, (float *)cellc, sigma_a, sigma_s, q, sc,
                           iso, dt, nsteps, s);
    } else {
        SnScat<double> sc{};
        for (int a = 0; a < KITRT_MAX_NMOM; ++a) sc.ga[a] = ga[a];
        rc = run_sn<double>(mn, quad_tab64(mn), (double *)psi, (double *)work, (double *)cellc, sigma_a, sigma_s, q,
                            sc, iso, dt, nsteps, s);
    }
    if (captured) return cudaFreeAsync(cellc, s) != cudaSuccess && !rc ? KITRT_ECUDA : rc;
    if (cudaEventRecord(mn->sn_done, s) != cudaSuccess) return rc ? rc : KITRT_ECUDA;
    mn->sn_pending = true;
    mn->sn_stream = id;
    return rc;
}

}  // extern "C"
