// Learned entropy closure: the MLP's alpha_{1..n-1}, the exact mass constraint for alpha_0, the
// FP64 moment-residual test and the hand-over of failing cells to Newton; plus the generator of
// training moments (von Mises-Fisher mixtures integrated with the solver's own quadrature).
//
// Mass constraint [Sec. 3.1: the ansatz must reproduce u; its zeroth moment is the particle
// density]: with z'_q = sum_{a>=1} alpha_a m_a(q) and U'_a = sum_q w_q exp(z'_q) m_a(q), the
// choice exp(alpha_0 m_0) = u_0 / U'_0 makes the zeroth moment of exp(alpha.m) equal to u_0, and
// every other moment is U_a = (u_0 / U'_0) U'_a. The cell keeps the network's answer when
// ||U - u||_2 <= fallback_tol ||u||_2 (computed in FP64); otherwise Newton starts from the better
// (by dual objective) of that point and the previous closure's, the latter with a step from its
// stored factor when the cell has one.
#include <cuda_bf16.h>
#include <math.h>

#include "kexp.cuh"
#include "kitrt_internal.cuh"
#include "newton_common.cuh"

namespace {

using namespace kitrt_dev;
constexpr int kWarps = 8;  // of the moment generator

// The network's points of the listed cells (S.list[1]): U'_a and the ansatz exp(z') of every point, in
// the fixed-point form of the sweeps (sweep.cuh). One thread per listed cell, work items (tile of 128
// cells, part of the quadrature) as in the FP64-mode sweep. A warp per cell in FP64 (28 FP64
// instructions a point for M_3) took, with the decision below and the network, 1.06 ms for 76,564
// M_3 closures of 400 points; now 0.30 ms.
constexpr int kSweepThreads = 128;

size_t learned_smem(int n, int N, int J) { return 2048 * 8 + (size_t)n * kSweepThreads * 8 + (size_t)J * 2 * N * 8; }

template <int NN>
__global__ void __launch_bounds__(kSweepThreads)
learned_sweep_kernel(Tables T, NewtonState S, const double *__restrict__ alpha_nn, double *__restrict__ Vacc, int vs,
                     int target_items, float *__restrict__ psi32)
{
    constexpr int n = Dims<NN>::n;
    extern __shared__ __align__(16) unsigned char learned_smem_raw[];
    uint64_t *tab = (uint64_t *)learned_smem_raw;
    int2 *sA = (int2 *)(tab + 2048);
    int2 *trig = sA + n * kSweepThreads;
    const int cnt = S.cnt[8], nunits = T.Qs / 32;
    const SweepSplit sp = sweep_split(cnt, gridDim.x, target_items, nunits);
    const int items = sp.tiles * sp.parts;
    if ((int)blockIdx.x >= items) return;
    for (int j = threadIdx.x; j < 2048; j += kSweepThreads) tab[j] = T.fx_exp[j];
    for (int j = threadIdx.x; j < T.J * 2 * NN; j += kSweepThreads) {
        const int p = j / (2 * NN), q = j % (2 * NN);
        trig[j] = T.fx_trig[p * 4 * NN + (q < NN ? q : NN + q)];
    }
    __syncthreads();
    int2 *myA = sA + threadIdx.x;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int tile = item / sp.parts, part = item % sp.parts;
        const int slot = tile * kSweepThreads + threadIdx.x;
        if (slot >= cnt) continue;  // threads are independent: no block barrier below
        const int q_begin = part * nunits / sp.parts * 8;
        const int q_end = min(T.nquad, (part + 1) * nunits / sp.parts * 8);
        const int cell = S.list[1][slot];
        const double *al = alpha_nn + (size_t)cell * n;  // al[0] = 0: alpha_0 follows from the mass
        float bound = 0.0f;
#pragma unroll
        for (int a = 0; a < n; ++a) {
            const double x = a ? al[a] : 0.0;
            const Limb w = kitrt_fx::split<32>(kitrt_fx::fx_from_double(x));
            myA[a * kSweepThreads] = make_int2(w.h, w.l);
            bound = fmaf(fabsf(d2f_bits(x)), T.fx_mmax[a], bound);
        }
        const int sh = fx_row_shift(bound);  // outside the range: scaled down; beyond that (-1) in FP64
        if (sh > 0) fx_scale_limbs(al, al, 0.0, 0, 1, n, sh, myA, kSweepThreads);  // al[0] = 0
        bool bad = false;
        long long U[n], A0 = 0;
#pragma unroll
        for (int c = 0; c < n; ++c) U[c] = 0;
        Limb A[2 * NN];
        FxSums<NN> B;
        B.clear();
        B.Sx = 100000;  // the first quad decides
        auto trial = [&](int a) {
            const int2 v = myA[a * kSweepThreads];
            return Limb{v.x, v.y};
        };
        auto moment = [&](int c) -> long long & { return U[c]; };
        int ring = q_begin / T.J, jq = q_begin - ring * T.J;
        bool fresh = true;
#pragma unroll 1
        for (int qd = q_begin; qd < q_end; ++qd) {
            if (fresh) {
                fx_coeffs<NN>(trial, T.fx_ringA + (size_t)ring * n, A0, A);
                fresh = false;
            }
            const int2 *tr = trig + jq * 2 * NN;
            const int pa = quad_pair0(ring, jq, T.P), pb = quad_pair1(ring, jq, T.P);
            Exp e[4];
            long long s[4];
            fx_exponents<NN>(A0, A, tr, NN, jq == 0, s);
            if (sh != 0) bad = !fx_outside_quad<NN>(sh, T, point_of(S, alpha_nn), cell, pa, pb, s) || bad;
#pragma unroll
            for (int t = 0; t < 4; ++t) e[t] = kitrt_fx::fx_exp(s[t], tab);
            if (psi32) {
                float *row = psi32 + (size_t)cell * T.Qp;
                float f[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) f[t] = __uint_as_float(kitrt_fx::fx_float_bits(e[t]));
                *(float2 *)(row + 2 * pa) = make_float2(f[0], f[1]);
                if (pb >= 0) *(float2 *)(row + 2 * pb) = make_float2(f[2], f[3]);
            }
            if (pb < 0) e[2] = e[3] = Exp{0, -100000};
            fx_accumulate<NN>(e, tr, NN, jq == 0, qd == q_begin, B, [&](int d) {
#pragma unroll
                for (int c = 0; c < n; ++c) U[c] = kitrt_fx::sar(U[c], d);
            });
            if (++jq == T.J) {
                fx_flush<NN>(T.fx_ringW + (size_t)ring * Dims<NN>::n2, T.fx_sumshift, B, moment);
                jq = 0;
                ++ring;
                fresh = true;
            }
        }
        if (!fresh) fx_flush<NN>(T.fx_ringW + (size_t)ring * Dims<NN>::n2, T.fx_sumshift, B, moment);
        double *col = Vacc + (size_t)part * cnt + slot;
        const int unit = fx_unit(B.Sx, T);
#pragma unroll
        for (int c = 0; c < n; ++c)
            col[(size_t)c * vs] = bad ? __longlong_as_double(0x7ff8000000000000LL) : kitrt_fx::fx_to_double(U[c], unit);
    }
}

// The decision per listed cell, one thread each: the network's point is kept, or Newton starts from it
// (an evaluation), or from the previous closure's point: with an evaluation, or, when its moments and
// a factor of the cell are stored, with the predictor's step (list S.handed[0], counter cnt[15]).
template <int NN>
__global__ void __launch_bounds__(64)
learned_decide_kernel(Tables T, NewtonState S, const double *__restrict__ u, const double *__restrict__ alpha_nn,
                      const double *__restrict__ Vacc, int vs, int sweep_grid, int target_items, double tol,
                      float *__restrict__ psi32, int first)
{
    constexpr int n = Dims<NN>::n;
    const int cnt = S.cnt[8], lane = threadIdx.x & 31;
    const int parts = sweep_split(cnt, sweep_grid, target_items, T.Qs / 32).parts;
    const int rounds = (cnt + gridDim.x * blockDim.x - 1) / (gridDim.x * blockDim.x);
    for (int rd = 0; rd < rounds; ++rd) {
        const int it = (rd * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
        const bool live = it < cnt;
        bool ok = false, to_eval = false, to_predict = false;
        int cell = 0;
        double c = 1.0;
        if (live) {
            cell = S.list[1][it];
            const size_t off = (size_t)cell * n;
            auto moment = [&](int a) {
                const double *col = Vacc + (size_t)a * vs + it;
                double v = col[0];
                for (int p = 1; p < parts; ++p) v += col[(size_t)p * cnt];
                return v;
            };
            const double u0 = u[off];
            c = u0 / moment(0);                       // exp(alpha_0 m_0)
            const double alpha0 = log(c) / T.m0;
            // residual and dual objective of the mass-corrected ansatz (<exp(alpha.m)> = u_0 / m_0)
            double r2 = 0.0, un2 = u0 * u0, au = alpha0 * u0, au_prev = first != 1 ? S.alpha[off] * u0 : 0.0;
#pragma unroll 1
            for (int a = 1; a < n; ++a) {
                const double ua = u[off + a], U = c * moment(a), r = U - ua;
                r2 = fma(r, r, r2);
                un2 = fma(ua, ua, un2);
                au = fma(alpha_nn[off + a], ua, au);
                if (first != 1) au_prev = fma(S.alpha[off + a], ua, au_prev);
            }
            const double f_nn = u0 / T.m0 - au;
            const bool finite = isfinite(alpha0) && isfinite(r2) && isfinite(f_nn) && u0 > 0.0;
            ok = finite && r2 <= tol * tol * un2;
            bool use_nn = finite;
            if (!ok && first != 1 && finite) {
                // the better start by dual objective (<exp> of the previous point is stored)
                const double f_prev = S.fsum[cell] - au_prev;
                use_nn = !(isfinite(f_prev) && f_prev <= f_nn);
            }
            if (ok || use_nn) {
                S.alpha[off] = alpha0;
#pragma unroll 1
                for (int a = 1; a < n; ++a) S.alpha[off + a] = alpha_nn[off + a];
            }
            if (ok) {
                S.U[off] = u0;
#pragma unroll 1
                for (int a = 1; a < n; ++a) S.U[off + a] = c * moment(a);
                S.fsum[cell] = u0 / T.m0;
                S.phase[cell] = PH_DONE;
            } else if (!use_nn && first != 1 && S.lfac && S.lfac[cell] && isfinite(S.fsum[cell])) {
                // (a cold cell's <exp> is poisoned: its stored moments and factor belong to another alpha)
                to_predict = true;
            } else {
                S.phase[cell] = PH_INIT;
                to_eval = true;
            }
        }
        // accepted cells: the ansatz takes the mass correction (a row at a time by the whole warp)
        unsigned rows = __ballot_sync(kFull, ok && psi32);
        while (rows) {
            const int src = __ffs(rows) - 1;
            rows &= rows - 1;
            const int rc = __shfl_sync(kFull, cell, src);
            const float cf = (float)__shfl_sync(kFull, c, src);
            for (int q = lane; q < T.Qp; q += 32) psi32[(size_t)rc * T.Qp + q] *= cf;
        }
        const unsigned nlive = __popc(__ballot_sync(kFull, live)), nfall = __popc(__ballot_sync(kFull, to_eval || to_predict)),
                       npred = __popc(__ballot_sync(kFull, to_predict));
        if (lane == 0) {
            if (nlive) atomicAdd(&S.cnt[10], (int)nlive);  // quadrature passes of the network's points
            if (nfall) atomicAdd(&S.cnt[5], (int)nfall);
            if (npred) atomicAdd(&S.cnt[9], (int)npred);   // steps from the stored factor
        }
        push_agg(S.list[0], &S.cnt[0], cell, to_eval);
        push_agg(S.handed[0], &S.cnt[15], cell, to_predict);
    }
}

// Moments of mixtures of von Mises-Fisher densities on S^2 on the folded rule: each folded point
// stands for the pair (Omega_2D, +-mu), and the basis is even in mu, so the pair contributes
// w/2 (f(mu) + f(-mu)) m. f(x) = sum_l weight_l kappa_l / (2 pi (1 - exp(-2 kappa_l)))
// exp(kappa_l (c_l . x - 1)). One warp per sample.
__global__ void vmf_moments_kernel(Tables T, const double *__restrict__ centres, const double *__restrict__ kappa,
                                   const double *__restrict__ weight, int lobes, int count,
                                   double *__restrict__ uout)
{
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int n = T.n, Qp = T.Qp;
    for (int s = blockIdx.x * kWarps + wib; s < count; s += gridDim.x * kWarps) {
        double acc[21];
        for (int a = 0; a < n; ++a) acc[a] = 0.0;
        for (int q = lane; q < T.Qf; q += 32) {
            const double wx = T.wox[q], wy = T.woy[q], w = T.w[q];
            const double ox = w > 0 ? wx / w : 0.0, oy = w > 0 ? wy / w : 0.0;
            const double mu = sqrt(fmax(0.0, 1.0 - ox * ox - oy * oy));
            double f = 0.0;
            for (int l = 0; l < lobes; ++l) {
                const double *cc = centres + ((size_t)s * lobes + l) * 3;
                const double k = kappa[(size_t)s * lobes + l], wt = weight[(size_t)s * lobes + l];
                if (wt == 0.0) continue;
                const double nrm = k / (2.0 * 3.14159265358979323846 * (1.0 - exp(-2.0 * k)));
                const double dp = cc[0] * ox + cc[1] * oy;
                f += wt * nrm * 0.5 * (exp(k * (dp + cc[2] * mu - 1.0)) + exp(k * (dp - cc[2] * mu - 1.0)));
            }
            for (int a = 0; a < n; ++a) acc[a] = fma(w * f, T.Mt[a * Qp + q], acc[a]);
        }
        for (int a = 0; a < n; ++a) {
            const double v = warp_sum(acc[a]);
            if (lane == 0) uout[(size_t)s * n + a] = v;
        }
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ x, __nv_bfloat16 *__restrict__ y, int P)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < P; k += gridDim.x * blockDim.x)
        y[k] = __float2bfloat16_rn(x[k]);
}

}  // namespace

int launch_learned_pass(kitrt_mn *mn, const Tables &T, const NewtonState &S, int C, const double *u,
                        NewtonParams np, float *psi32, int first, cudaStream_t s)
{
    const size_t smem = learned_smem(mn->n, mn->N, mn->J);
    int blocks = (C + 63) / 64;
    if (blocks > mn->nsm * 16) blocks = mn->nsm * 16;
    if (blocks < 1) blocks = 1;
    {
        LaunchScope ls(mn, PK_MLP, s, 0);
        mn->launch_count += 1;  // two kernels in this scope
#define LP_CASE(NNv)                                                                                       \
    case NNv:                                                                                              \
        if (ensure_dyn_smem(learned_sweep_kernel<NNv>, smem)) return KITRT_ECUDA;                          \
        learned_sweep_kernel<NNv><<<mn->grid_fp64, kSweepThreads, smem, s>>>(T, S, mn->d_alpha_nn, mn->d_Vacc, mn->vs, \
                                                                             mn->target_fp64, psi32);      \
        learned_decide_kernel<NNv><<<blocks, 64, 0, s>>>(T, S, u, mn->d_alpha_nn, mn->d_Vacc, mn->vs, mn->grid_fp64,   \
                                                         mn->target_fp64, mn->p.fallback_tol, psi32, first); \
        break;
        switch (mn->N) {
            LP_CASE(1)
            LP_CASE(2)
            LP_CASE(3)
            LP_CASE(4)
            LP_CASE(5)
        default: return KITRT_EINVAL;
        }
#undef LP_CASE
        if (cudaGetLastError() != cudaSuccess) return KITRT_ECUDA;
    }
    if (first == 1) return KITRT_OK;
    return launch_predict(mn, S, C, u, np, S.handed[0], S.cnt + 15, s);
}

extern "C" {

int32_t kitrt_mn_set_mlp(kitrt_mn *mn, const float *params, const float *norm, int32_t hidden, void *stream)
{
    if (!mn || !params || !norm || hidden != 64) return KITRT_EINVAL;
    const int dio = mn->n - 1;
    const int P = kitrt_mlp_param_count(dio, hidden, dio);
    cudaStream_t s = (cudaStream_t)stream;
    if (!mn->d_mlp16) {
        if (cudaMalloc(&mn->d_mlp16, sizeof(uint16_t) * P) != cudaSuccess) return KITRT_ENOMEM;
        mn->allocs.push_back(mn->d_mlp16);
        if (cudaMalloc(&mn->d_mlp_norm, sizeof(float) * 4 * dio) != cudaSuccess) return KITRT_ENOMEM;
        mn->allocs.push_back(mn->d_mlp_norm);
    }
    to_bf16_kernel<<<(P + 255) / 256, 256, 0, s>>>(params, (__nv_bfloat16 *)mn->d_mlp16, P);
    if (cudaMemcpyAsync(mn->d_mlp_norm, norm, sizeof(float) * 4 * dio, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return KITRT_ECUDA;
    mn->has_mlp = true;
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int32_t kitrt_vmf_moments(kitrt_mn *mn, const double *centres, const double *kappa, const double *weight,
                          int32_t lobes, int32_t count, double *u, void *stream)
{
    if (!mn || !centres || !kappa || !weight || !u || lobes < 1 || count < 0) return KITRT_EINVAL;
    if (count == 0) return KITRT_OK;
    int blocks = (count + kWarps - 1) / kWarps;
    if (blocks > mn->nsm * 16) blocks = mn->nsm * 16;
    vmf_moments_kernel<<<blocks, kWarps * 32, 0, (cudaStream_t)stream>>>(mn->tables(), centres, kappa, weight, lobes,
                                                                         count, u);
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

}  // extern "C"
