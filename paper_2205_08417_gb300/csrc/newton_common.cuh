// Device helpers shared by the closure kernels: warp reductions, the warp Cholesky factorisation
// and solves, and the per-cell Newton logic that follows one evaluation of the dual
// [Sec. 3.1, Eq. entropyOCP: dual f(alpha) = <exp(alpha.m)> - alpha.u, gradient <m e> - u,
// Hessian <m m^T e>], with Armijo backtracking.
#pragma once

#include <math.h>

#include "kitrt_internal.cuh"
#include "sweep.cuh"

namespace kitrt_dev {

constexpr unsigned kFull = 0xffffffffu;
// (1e-14)^2: residuals below 1e-14 ||u|| need no further Newton or polish step
constexpr double kRoundoff2 = 1e-28;
// mixed Hessian: a Newton step that does not halve the residual sends the cell to FP64
constexpr double kStallRatio = 0.5;

template <int NN>
struct Dims {
    static constexpr int n = (NN + 1) * (NN + 2) / 2;
    static constexpr int n2 = (2 * NN + 1) * (2 * NN + 2) / 2;
    static constexpr int npairs = n * (n + 1) / 2;
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ void push(int32_t *list, int32_t *cnt, int cell, int lane)
{
    if (lane == 0) {
        int pos = atomicAdd(cnt, 1);
        list[pos] = cell;
    }
}

// A mixed-mode cell goes over to the FP64 Hessian (FP64 sweep) from the next round on; counted
// once per cell and closure (S.cnt[11]).
__device__ __forceinline__ void hand_over(const NewtonState &S, int cell)
{
    if (!S.h64[cell]) {
        S.h64[cell] = 1;
        atomicAdd(&S.cnt[11], 1);
    }
}

__device__ __forceinline__ void fail(const NewtonState &S, int cell, int code, int lane)
{
    if (lane == 0) {
        S.status[cell] = code;
        S.phase[cell] = PH_DONE;
        atomicAdd(&S.cnt[3], 1);
    }
}

// Packed lower-triangle index of (a, b), b <= a.
__device__ __forceinline__ int tri_idx(int a, int b) { return a * (a + 1) / 2 + b; }

// Warp Cholesky of the n x n matrix in sH (row-major). On success the strict lower triangle
// holds L and the diagonal holds 1/L_jj, so the triangular solves multiply instead of divide
// (FP64 division costs many FP64-pipe instructions).
template <int n>
__device__ bool warp_cholesky(double *sH, int lane)
{
    for (int j = 0; j < n; ++j) {
        const double djj = sH[j * n + j];
        if (!(djj > 0.0)) return false;  // warp-uniform: every lane read the same value
        const double rinv = 1.0 / sqrt(djj);
        __syncwarp();
        if (lane > j && lane < n) sH[lane * n + j] *= rinv;
        if (lane == j) sH[j * n + j] = rinv;
        __syncwarp();
        if (lane > j && lane < n) {
            const double lij = sH[lane * n + j];
            for (int k = j + 1; k <= lane; ++k) sH[lane * n + k] = fma(-lij, sH[k * n + j], sH[lane * n + k]);
        }
        __syncwarp();
    }
    return true;
}

// Solve L L^T x = b (factor from warp_cholesky, inverse diagonal) with lane a holding b_a;
// returns x_a in lane a.
template <int n>
__device__ double warp_chol_solve(const double *sH, double b, int lane)
{
    double y = b;
    for (int j = 0; j < n; ++j) {
        const double yj = __shfl_sync(kFull, y, j) * sH[j * n + j];
        if (lane == j) y = yj;
        if (lane > j && lane < n) y = fma(-sH[lane * n + j], yj, y);
    }
    for (int j = n - 1; j >= 0; --j) {
        const double xj = __shfl_sync(kFull, y, j) * sH[j * n + j];
        if (lane == j) y = xj;
        if (lane < j) y = fma(-sH[j * n + lane], xj, y);
    }
    return lane < n ? y : 0.0;
}

// Newton logic of one cell after an evaluation of the dual at the trial point `at` (lane a holds
// component a). Vs holds the n2 degree-2N moments sum_q w_q e_q m~_c(q) (warp-visible), whose
// first n entries are the ansatz moments U. One warp per cell; every branch is warp-uniform. Used by the
// allocation-free closure, in FP64 throughout.
template <int NN>
__device__ void newton_post(const Tables &T, const NewtonState &S, const NewtonParams &np,
                            int cell, int ph, double lam, double at, double ua, const double *Vs,
                            double *H, int32_t *list_out, int32_t *cnt_out, int lane)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, npairs = Dims<NN>::npairs;
    const size_t off = (size_t)cell * n;
    bool finite = true;
    for (int c = 0; c < n2; ++c) finite = finite && isfinite(Vs[c]);
    const double fs = Vs[0] / T.m0;
    const double au = warp_sum(at * ua);
    const double ar2 = warp_sum(lane < n && lane >= np.reg0 ? at * at : 0.0);
    const double ft = fma(0.5 * np.gamma, ar2, fs - au);
    if (lane == 0) {
        const int ev = S.evals[cell] + 1;
        S.evals[cell] = ev;
        atomicMax(&S.cnt[4], ev);
        atomicAdd(&S.cnt[6], 1);
    }
    bool accept;
    if (ph == PH_INIT) {
        if (!finite) {
            fail(S, cell, KITRT_ENOTREALIZABLE, lane);
            return;
        }
        accept = true;
    } else {
        const double fs0 = S.fsum[cell], f0 = S.f0[cell];
        const double slack = 64.0 * 2.220446049250313e-16 * (fs0 + fabs(fs0 - f0));
        accept = finite && ft <= f0 + np.c1 * lam * S.gd[cell] + slack;
    }
    if (!accept) {
        const int h = S.halv[cell] + 1;
        if (h > np.max_halvings) {
            fail(S, cell, KITRT_ELINESEARCH, lane);
        } else {
            if (lane == 0) {
                S.halv[cell] = h;
                S.lam[cell] = 0.5 * lam;
            }
            push(list_out, cnt_out, cell, lane);
        }
        return;
    }
    // Hessian H_ab = sum_c G_abc V_c from the Gaunt coefficients
    for (int p = lane; p < npairs; p += 32) {
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= p) ++a;
        const int b = p - a * (a + 1) / 2;
        double h = 0.0;
        for (int t = T.gstart[p]; t < T.gstart[p + 1]; ++t) h = fma(T.gcoef[t], Vs[T.gidx[t]], h);
        if (a == b && a >= np.reg0) h += np.gamma;  // regularized moments
        H[a * n + b] = h;
        H[b * n + a] = h;
    }
    __syncwarp();
    if (!warp_cholesky<n>(H, lane)) {
        __syncwarp();
        fail(S, cell, KITRT_ECHOL, lane);
        return;
    }
    // accepted: store the point, its moments and the factor of H
    const double Ua = lane < n ? Vs[lane] : 0.0;
    if (lane < n) {
        S.alpha[off + lane] = at;
        S.U[off + lane] = Ua;
    }
    if (lane == 0) {
        S.fsum[cell] = fs;
        S.f0[cell] = ft;
    }
    for (int a = lane; a < n; a += 32)
        for (int b = 0; b <= a; ++b) S.L[(size_t)cell * npairs + tri_idx(a, b)] = H[a * n + b];
    const double g = lane < n ? fma(lane >= np.reg0 ? np.gamma : 0.0, at, Ua - ua) : 0.0;
    const double d = warp_chol_solve<n>(H, -g, lane);
    __syncwarp();
    const double gn2 = warp_sum(g * g), un2 = warp_sum(ua * ua), gd = warp_sum(g * d);
    if (lane < n) S.dir[off + lane] = d;
    int iters = S.iters[cell];
    if (ph == PH_NEWTON) ++iters;
    if (lane == 0) S.iters[cell] = iters;
    if (gn2 <= np.tau * np.tau * un2) {
        if (lane == 0) S.phase[cell] = PH_DONE;
        return;
    }
    if (iters >= np.max_iter) {
        fail(S, cell, KITRT_ENOCONVERGE, lane);
        return;
    }
    if (lane == 0) {
        S.gd[cell] = gd;
        S.lam[cell] = 1.0;
        S.halv[cell] = 0;
        S.phase[cell] = PH_NEWTON;
    }
    push(list_out, cnt_out, cell, lane);
}

}  // namespace kitrt_dev

namespace kitrt_dev {

// Warp-aggregated append of `cell` to a list when pred holds (all active lanes must call it).
// Returns the cell's position in the list.
__device__ __forceinline__ int push_agg(int32_t *list, int32_t *cnt, int cell, bool pred)
{
    const unsigned act = __activemask();
    const unsigned m = __ballot_sync(act, pred);
    if (!m) return 0;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(act, base, leader);
    const int at = base + __popc(m & ((1u << lane) - 1u));
    if (pred) list[at] = cell;
    return at;
}

__device__ __forceinline__ float r_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ bool r_pos(float d) { return d > 0.0f && d < 3.0e38f; }
__device__ __forceinline__ bool r_pos(double d) { return d > 0.0; }
__device__ __forceinline__ float r_rsqrt(float a) { return rsqrtf(a); }
// 1/sqrt(a): the FP32 value improved by one third-order step y (1 + e/2 + 3 e^2 / 8), e = 1 - a y^2
// (the binomial series of (1 - e)^(-1/2); e is about 1e-7, the dropped term 1e-22), five FP64
// instructions; outside the float range the library function.
static __device__ __noinline__ double r_rsqrt_any(double a) { return rsqrt(a); }
__device__ __forceinline__ double r_rsqrt(double a)
{
    if (!(a > 1e-37 && a < 1e37)) return r_rsqrt_any(a);
    const double y = f2d_bits(rsqrtf(d2f_bits(a)));
    const double e = fma(-a * y, y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// Newton step of one listed cell after a round of sweeps, in the FP64 mode for N <= 3 when many
// cells are listed (launch_post): one thread per cell, so that every FP64 instruction works for 32
// cells. The Hessian assembly, the Cholesky factorisation and the two triangular solves run as
// rolled loops over per-thread slices of shared memory (entry e of a thread at e * B + thread):
// fully unrolled code (several thousand instructions, run once) waited mostly on instruction fetch
// (ncu: stalls on no_instruction ~3x those on memory).

// H (packed lower, + gamma on the regularized diagonal) from the Gaunt terms, its Cholesky factor
// (1/L_jj on the diagonal) in place, then y <- -H^-1 y in place. V: the moments, entry c at V[c B];
// entry e of L and y at e B. Returns false when the factorisation breaks down.
template <int NN>
__device__ bool hess_factor_solve(const Tables &T, const NewtonParams &np, const double *V, double *L, double *y, int B)
{
    constexpr int n = Dims<NN>::n, npairs = Dims<NN>::npairs;
#pragma unroll 1
    for (int p = 0; p < npairs; ++p) {
        double h = 0.0;
        const int t1 = T.gstart[p + 1];
#pragma unroll 1
        for (int t = T.gstart[p]; t < t1; ++t) h = fma(T.gcoef[t], V[(size_t)T.gidx[t] * B], h);
        L[(size_t)p * B] = h;
    }
    if (np.gamma != 0.0) {
#pragma unroll 1
        for (int j = np.reg0; j < n; ++j) L[(size_t)tri_idx(j, j) * B] += np.gamma;
    }
    bool spd = true;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const int jj = j * (j + 1) / 2;
        double d = L[(size_t)(jj + j) * B];
#pragma unroll 1
        for (int k = 0; k < j; ++k) {
            const double l = L[(size_t)(jj + k) * B];
            d = fma(-l, l, d);
        }
        spd = spd && d > 0.0;
        const double rinv = r_rsqrt(d > 0.0 ? d : 1.0);
        L[(size_t)(jj + j) * B] = rinv;
#pragma unroll 1
        for (int i = j + 1; i < n; ++i) {
            const int ii = i * (i + 1) / 2;
            double sacc = L[(size_t)(ii + j) * B];
#pragma unroll 1
            for (int k = 0; k < j; ++k)
                sacc = fma(-L[(size_t)(ii + k) * B], L[(size_t)(jj + k) * B], sacc);
            L[(size_t)(ii + j) * B] = sacc * rinv;
        }
    }
    if (!spd) return false;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const int ii = i * (i + 1) / 2;
        double sacc = y[(size_t)i * B];
#pragma unroll 1
        for (int k = 0; k < i; ++k) sacc = fma(-L[(size_t)(ii + k) * B], y[(size_t)k * B], sacc);
        y[(size_t)i * B] = sacc * L[(size_t)(ii + i) * B];
    }
#pragma unroll 1
    for (int i = n - 1; i >= 0; --i) {
        double sacc = y[(size_t)i * B];
#pragma unroll 1
        for (int k = i + 1; k < n; ++k) sacc = fma(-L[(size_t)tri_idx(k, i) * B], y[(size_t)k * B], sacc);
        y[(size_t)i * B] = sacc * L[(size_t)tri_idx(i, i) * B];
    }
    return true;
}

// V: the cell's moments; Lsm, ysm: this thread's columns of [npairs x B] and [n x B] doubles.
// Returns true when the cell continues (must be appended to the next list).
template <int NN>
__device__ bool newton_cell(const Tables &T, const NewtonState &S, const NewtonParams &np, int cell,
                            const double *__restrict__ V, double *Lsm, double *ysm, int B,
                            const double *__restrict__ u, int &evals_out)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, npairs = Dims<NN>::npairs;
    const size_t off = (size_t)cell * n;
    const int ph = S.phase[cell];
    const double lam = ph == PH_NEWTON ? S.lam[cell] : 0.0;
    const bool reg = np.gamma != 0.0;
    double at[n], ua[n];
    double au = 0.0, ar2 = 0.0;
#pragma unroll
    for (int a = 0; a < n; ++a) {
        const double al = S.alpha[off + a];
        at[a] = ph == PH_NEWTON ? fma(lam, S.dir[off + a], al) : al;
        ua[a] = u[off + a];
        au = fma(at[a], ua[a], au);
        if (reg && a >= np.reg0) ar2 = fma(at[a], at[a], ar2);
    }
    bool finite = true;
#pragma unroll
    for (int c = 0; c < n2; ++c) finite = finite && finite_bits(V[(size_t)c * B]);
    const double fs = V[0] * T.rm0;
    const double ft = reg ? fma(0.5 * np.gamma, ar2, fs - au) : fs - au;
    const int ev = S.evals[cell] + 1;
    S.evals[cell] = ev;
    evals_out = ev;
    auto fail_t = [&](int code) {
        S.status[cell] = code;
        S.phase[cell] = PH_DONE;
        atomicAdd(&S.cnt[3], 1);
    };
    bool accept;
    if (ph == PH_INIT) {
        if (!finite) {
            fail_t(KITRT_ENOTREALIZABLE);
            return false;
        }
        accept = true;
    } else {
        const double fs0 = S.fsum[cell], f0 = S.f0[cell];
        const double slack = 64.0 * 2.220446049250313e-16 * (fs0 + fabs(fs0 - f0));
        accept = finite && ft <= f0 + np.c1 * lam * S.gd[cell] + slack;
    }
    if (!accept) {
        const int h = S.halv[cell] + 1;
        if (h > np.max_halvings) {
            fail_t(KITRT_ELINESEARCH);
            return false;
        }
        S.halv[cell] = h;
        S.lam[cell] = 0.5 * lam;
        return true;
    }
    double g[n], y[n];
#pragma unroll
    for (int a = 0; a < n; ++a) {
        g[a] = V[(size_t)a * B] - ua[a];
        if (reg && a >= np.reg0) g[a] = fma(np.gamma, at[a], g[a]);
        ysm[(size_t)a * B] = -g[a];
    }
    if (!hess_factor_solve<NN>(T, np, V, Lsm, ysm, B)) {
        fail_t(KITRT_ECHOL);
        return false;
    }
#pragma unroll
    for (int a = 0; a < n; ++a) y[a] = ysm[(size_t)a * B];
#pragma unroll 1
    for (int p = 0; p < npairs; ++p) S.L[(size_t)cell * npairs + p] = Lsm[(size_t)p * B];
#pragma unroll
    for (int a = 0; a < n; ++a) {
        S.alpha[off + a] = at[a];
        S.U[off + a] = V[(size_t)a * B];
    }
    S.fsum[cell] = fs;
    S.f0[cell] = ft;
    double gn2 = 0.0, un2 = 0.0, gd = 0.0;
#pragma unroll
    for (int a = 0; a < n; ++a) {
        gn2 = fma(g[a], g[a], gn2);
        un2 = fma(ua[a], ua[a], un2);
        gd = fma(g[a], y[a], gd);
        S.dir[off + a] = y[a];
    }
    int iters = S.iters[cell];
    if (ph == PH_NEWTON) ++iters;
    S.iters[cell] = iters;
    if (gn2 <= np.tau * np.tau * un2) {
        S.phase[cell] = PH_DONE;
        return false;
    }
    if (iters >= np.max_iter) {
        fail_t(KITRT_ENOCONVERGE);
        return false;
    }
    S.gd[cell] = gd;
    S.lam[cell] = 1.0;
    S.halv[cell] = 0;
    S.phase[cell] = PH_NEWTON;
    return true;
}

constexpr int kPostBlock = 64;

// Dynamic shared memory of post_thread_kernel: [n2 x kPostBlock], [npairs x kPostBlock] and
// [n x kPostBlock] doubles (moments, factor, solve vector), the Gaunt coefficients, the moment
// indices and the npairs + 1 term starts.
__host__ __device__ inline size_t post_smem_bytes(int n, int n2, int npairs, int nnz)
{
    return (size_t)(n2 + npairs + n) * kPostBlock * 8 + (size_t)nnz * 12 + (size_t)(npairs + 1) * 4;
}

// The listed cells, when more than `above` of them, one thread each; otherwise post_group_kernel takes
// the round. The sweeps' parts are added in order while the moments are loaded, which saves a launch
// and a pass a round (adjoint, 59,168 cells, 32 closures: 15.7 -> 15.0 ms with 1/sqrt by r_rsqrt).
template <int NN>
__global__ void __launch_bounds__(kPostBlock)
post_thread_kernel(Tables T, NewtonState S, const double *__restrict__ u, int k, NewtonParams np,
                   const double *__restrict__ Vacc, int vs, int nnz, int sweep_grid, int target_items, int nunits,
                   int above)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, npairs = Dims<NN>::npairs;
    extern __shared__ __align__(16) unsigned char post_smem[];
    double *sV = reinterpret_cast<double *>(post_smem);                     // [n2][thread]
    double *sL = sV + (size_t)n2 * kPostBlock;                              // [npairs][thread]
    double *sy = sL + (size_t)npairs * kPostBlock;                          // [n][thread]
    double *coef = sy + (size_t)n * kPostBlock;
    int32_t *gidx = reinterpret_cast<int32_t *>(coef + nnz);
    int32_t *gstart = gidx + nnz;
    const int32_t *list_in = S.list[k & 1];
    int32_t *list_out = S.list[(k + 1) & 1];
    const int cnt_in = S.cnt[k % 3];
    const int stride = gridDim.x * blockDim.x;
    // uniform: not this kernel's round, or this block has no slot
    if (cnt_in <= above || (int)(blockIdx.x * blockDim.x) >= cnt_in) return;
    const int parts = sweep_split(cnt_in, sweep_grid, target_items, nunits).parts;
    int32_t *cnt_out = &S.cnt[(k + 1) % 3];
    // stage the Gaunt tables and point this block's view of them at the copies
    for (int t = threadIdx.x; t < nnz; t += blockDim.x) {
        gidx[t] = T.gidx[t];
        coef[t] = T.gcoef[t];
    }
    for (int t = threadIdx.x; t <= npairs; t += blockDim.x) gstart[t] = T.gstart[t];
    __syncthreads();
    Tables Ts = T;
    Ts.gidx = gidx;
    Ts.gstart = gstart;
    Ts.gcoef = coef;
    const int rounds = (cnt_in + stride - 1) / stride;
    for (int rd = 0; rd < rounds; ++rd) {
        const int it = rd * stride + blockIdx.x * blockDim.x + threadIdx.x;
        bool cont = false;
        int cell = -1, ev = 0;
        if (it < cnt_in) {
            cell = list_in[it];
            double *mine = sV + threadIdx.x;
#pragma unroll
            for (int c = 0; c < n2; ++c) mine[c * kPostBlock] = Vacc[(size_t)c * vs + it];
            for (int p = 1; p < parts; ++p) {
                const double *col = Vacc + (size_t)p * cnt_in + it;
#pragma unroll
                for (int c = 0; c < n2; ++c) mine[c * kPostBlock] += col[(size_t)c * vs];
            }
            cont = newton_cell<NN>(Ts, S, np, cell, mine, sL + threadIdx.x, sy + threadIdx.x, kPostBlock, u, ev);
        }
        // every slot taken in this round is one evaluation
        const unsigned act = __activemask();
        const unsigned live = __ballot_sync(act, it < cnt_in);
        const int evmax = __reduce_max_sync(act, ev);
        if ((threadIdx.x & 31) == __ffs(act) - 1 && live) {
            atomicAdd(&S.cnt[6], __popc(live));
            atomicMax(&S.cnt[4], evmax);
        }
        push_agg(list_out, cnt_out, cell, cont);
    }
}

// ---------------------------------------------------------------------------------------------
// Newton step with 8 lanes per cell (every mixed-mode round; FP64 mode for N >= 4 or few cells).
//
// A round lists anything from a few hundred to all cells. One thread per cell leaves a serial chain
// of a few thousand dependent instructions, and its factor does not fit a thread's registers for
// N >= 4 (120 or 231 entries). Here 8 lanes share a cell: lane g owns the rows g, g + 8, g + 16 of
// the Hessian and its factor in registers, pivots and columns travel by shuffles, and the packed
// matrix passes through shared memory only to be assembled (entries dealt to the lanes) and to be
// written out in whole rows. Measured against the thread-per-cell kernels with their separate
// summation of the sweeps' parts (part of the load here), Newton time of a run: M_5, 996,872 cells,
// two steps 70.3 -> 13.7 ms; M_4, 20,000 cells 1.09 -> 0.21 ms; M_3, 99,458 cells, four steps
// 0.94 -> 0.68 ms (0.73 before each cell's state was read ahead of its moments); M_2 in FP64 mode,
// 3,872 cells 0.25 -> 0.17 ms.
// ---------------------------------------------------------------------------------------------
constexpr int kGroupBlock = 256;
constexpr int kGroupCells = kGroupBlock / 8;  // cells per block and pass
constexpr int kGroupPitch = kGroupCells + 1;  // row pitch of the moments in shared memory

__device__ __forceinline__ double group_sum(double v)
{
    v += __shfl_xor_sync(kFull, v, 4);
    v += __shfl_xor_sync(kFull, v, 2);
    v += __shfl_xor_sync(kFull, v, 1);
    return v;
}

// f(Int<B>) ... f(Int<E - 1>): a loop whose index is a compile-time constant
template <int I>
struct Int {
    __host__ __device__ constexpr operator int() const { return I; }
};
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F &&f)
{
    if constexpr (B < E) {
        f(Int<B>{});
        static_for<B + 1, E>(f);
    }
}

// Assembly, factorisation and solve of one cell per group, in precision R: H from the Gaunt terms
// (coef, idx; Vr: the block's moments in R, entry c of this cell at Vr[c kGroupPitch]) into Hs
// [npairs], its factor (1/L_jj on the diagonal) back into Hs, and y <- H^-1 y (row g + 8 s in y[s]).
// Whole warps; cells that do not take part compute along. Returns whether H was positive definite.
template <int NN, typename R, typename Coef, typename Idx>
__device__ __forceinline__ bool group_factor_solve(const Coef *__restrict__ coef, const Idx *__restrict__ idx,
                                                   const int32_t *__restrict__ gstart, const R *Vr, R *Hs,
                                                   R gamma, int reg0, int g, R (&y)[(Dims<NN>::n + 7) / 8])
{
    constexpr int n = Dims<NN>::n, npairs = Dims<NN>::npairs, SL = (n + 7) / 8;
    for (int p = g; p < npairs; p += 8) {
        R h = R(0);
        const int t1 = gstart[p + 1];
        for (int t = gstart[p]; t < t1; ++t) h = r_fma((R)coef[t], Vr[(int)idx[t] * kGroupPitch], h);
        Hs[p] = h;
    }
    __syncwarp();
    // row g + 8 s in r[s n ..] (columns beyond the row are not used); every index below is a
    // compile-time constant, so that the rows stay in registers
    R r[SL * n];
    static_for<0, SL>([&](auto S) {
        static_for<0, (8 * S + 8 < n ? 8 * S + 8 : n)>([&](auto K) {
            const int row = g + 8 * S;
            r[S * n + K] = row < n && K <= row ? Hs[row * (row + 1) / 2 + K] : R(0);
            if (K == row && row >= reg0) r[S * n + K] += gamma;
        });
    });
    bool spd = true;
    static_for<0, n>([&](auto J) {
        constexpr int j = J, sj = J / 8, own = sj * n + j;
        const R d = __shfl_sync(kFull, r[own], j & 7, 8);
        spd = spd && r_pos(d);
        const R rinv = r_rsqrt(d > R(0) ? d : R(1));
        static_for<sj, SL>([&](auto S) {
            const R scaled = r[S * n + j] * rinv;
            r[S * n + j] = g + 8 * S == j ? rinv : scaled;
        });
        static_for<j + 1, n>([&](auto K) {
            const R l = __shfl_sync(kFull, r[(K / 8) * n + j], K & 7, 8);
            static_for<K / 8, SL>([&](auto S) { r[S * n + K] = r_fma(-r[S * n + j], l, r[S * n + K]); });
        });
        // forward substitution with the finished column
        const R yj = __shfl_sync(kFull, y[sj] * r[own], j & 7, 8);
        static_for<sj, SL>([&](auto S) {
            const R next = r_fma(-r[S * n + j], yj, y[S]);
            y[S] = g + 8 * S == j ? yj : g + 8 * S > j ? next : y[S];
        });
    });
    __syncwarp();
    static_for<0, SL>([&](auto S) {
        static_for<0, (8 * S + 8 < n ? 8 * S + 8 : n)>([&](auto K) {
            const int row = g + 8 * S;
            if (row < n && K <= row) Hs[row * (row + 1) / 2 + K] = r[S * n + K];
        });
    });
    __syncwarp();
    // backward substitution: row j of the factor from shared memory
    static_for<0, n>([&](auto I) {
        constexpr int j = n - 1 - I, sj = j / 8;
        const R xj = __shfl_sync(kFull, y[sj] * r[sj * n + j], j & 7, 8);
        static_for<0, sj + 1>([&](auto S) {
            const int row = g + 8 * S;
            if (row < j) y[S] = r_fma(-Hs[j * (j + 1) / 2 + row], xj, y[S]);
            if (row == j) y[S] = xj;
        });
    });
    return spd;
}

// The same in FP64 with the matrix in shared memory throughout: the few cells of the mixed modes that
// were handed over to the FP64 Hessian. The register version would set the register count of the
// whole kernel (and with it how many blocks an SM holds) for cells that are mostly not there.
template <int NN>
__device__ __forceinline__ bool group_factor_solve_shared(const Tables &T, const double *V, double *Hs, double gamma,
                                                          int reg0, int g, double (&y)[(Dims<NN>::n + 7) / 8])
{
    constexpr int n = Dims<NN>::n, npairs = Dims<NN>::npairs, SL = (n + 7) / 8;
#pragma unroll 1
    for (int p = g; p < npairs; p += 8) {
        double h = 0.0;
        const int t1 = T.gstart[p + 1];
#pragma unroll 1
        for (int t = T.gstart[p]; t < t1; ++t) h = fma(T.gcoef[t], V[T.gidx[t] * kGroupPitch], h);
        Hs[p] = h;
    }
    __syncwarp();
#pragma unroll 1
    for (int j = reg0 + g; j < n; j += 8) Hs[tri_idx(j, j)] += gamma;
    __syncwarp();
    bool spd = true;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const double d = Hs[tri_idx(j, j)];
        spd = spd && r_pos(d);
        const double rinv = r_rsqrt(d > 0.0 ? d : 1.0);
        __syncwarp();
        if (g == 0) Hs[tri_idx(j, j)] = rinv;
#pragma unroll 1
        for (int i = j + 1 + g; i < n; i += 8) Hs[tri_idx(i, j)] *= rinv;
        __syncwarp();
#pragma unroll 1
        for (int i = j + 1 + g; i < n; i += 8) {
            const double l = Hs[tri_idx(i, j)];
#pragma unroll 1
            for (int k = j + 1; k <= i; ++k) Hs[tri_idx(i, k)] = fma(-l, Hs[tri_idx(k, j)], Hs[tri_idx(i, k)]);
        }
        __syncwarp();
    }
#pragma unroll
    for (int sj = 0; sj < SL; ++sj)
#pragma unroll 1
        for (int j = 8 * sj; j < (8 * sj + 8 < n ? 8 * sj + 8 : n); ++j) {
            const double yj = __shfl_sync(kFull, y[sj] * Hs[tri_idx(j, j)], j & 7, 8);
#pragma unroll
            for (int s = sj; s < SL; ++s) {
                const int row = g + 8 * s;
                if (row == j) y[s] = yj;
                else if (row > j && row < n) y[s] = fma(-Hs[tri_idx(row, j)], yj, y[s]);
            }
        }
#pragma unroll
    for (int sj = SL - 1; sj >= 0; --sj)
#pragma unroll 1
        for (int j = (8 * sj + 8 < n ? 8 * sj + 8 : n) - 1; j >= 8 * sj; --j) {
            const double xj = __shfl_sync(kFull, y[sj] * Hs[tri_idx(j, j)], j & 7, 8);
#pragma unroll
            for (int s = 0; s <= sj; ++s) {
                const int row = g + 8 * s;
                if (row == j) y[s] = xj;
                else if (row < j) y[s] = fma(-Hs[tri_idx(j, row)], xj, y[s]);
            }
        }
    return spd;
}

// Dynamic shared memory of post_group_kernel: moments [n2][pitch] (FP64, and FP32 in the mixed
// modes), one packed matrix per cell, the Gaunt coefficients of the mode, indices and starts, and
// the pass's cells.
__host__ __device__ inline size_t group_smem_bytes(int n2, int npairs, int nnz, bool mixed)
{
    return (size_t)n2 * kGroupPitch * (mixed ? 12 : 8) + (size_t)kGroupCells * npairs * 8 + (size_t)nnz * (mixed ? 4 : 8) +
           (size_t)((nnz + 3) / 4 * 4) + (size_t)(npairs + 1) * 4 + 2 * kGroupCells * 4 + 2 * kGroupCells * 8;
}

template <int NN, bool MIXED>
__global__ void __launch_bounds__(kGroupBlock, MIXED && NN <= 3 ? 3 : 2)
post_group_kernel(Tables T, NewtonState S, const double *__restrict__ u, int k, NewtonParams np,
                  const double *__restrict__ Vacc, int vs, int vs_handed, int nnz, int sweep_grid, int target_items,
                  int nunits, int grid64, int target64, int nunits64, int upto)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, npairs = Dims<NN>::npairs, SL = (n + 7) / 8;
    extern __shared__ __align__(16) unsigned char group_smem[];
    double *sV = reinterpret_cast<double *>(group_smem);                           // [n2][pitch]
    double *sH = sV + n2 * kGroupPitch;                                            // [cell][npairs]
    double *sAu = sH + kGroupCells * npairs;                                       // [2][cell]
    unsigned char *coef = reinterpret_cast<unsigned char *>(sAu + 2 * kGroupCells);
    float *sVf = reinterpret_cast<float *>(coef + (size_t)nnz * (MIXED ? 4 : 8));  // [n2][pitch]
    int32_t *gstart = reinterpret_cast<int32_t *>(sVf + (MIXED ? n2 * kGroupPitch : 0));
    int32_t *scell = gstart + npairs + 1, *sh64 = scell + kGroupCells;
    unsigned char *gidx = reinterpret_cast<unsigned char *>(sh64 + kGroupCells);
    const int32_t *list_in = S.list[k & 1];
    int32_t *list_out = S.list[(k + 1) & 1];
    const int cnt_in = S.cnt[k % 3];
    // uniform: not this kernel's round, or no slot for this block
    if (cnt_in > upto || (int)blockIdx.x * kGroupCells >= cnt_in) return;
    const int parts = sweep_split(cnt_in, sweep_grid, target_items, nunits).parts;
    // handed cells: split on their own, the parts after the first from column vs_handed on
    const int handed = MIXED ? S.cnt[12 + k % 3] : 0;
    const int parts64 = MIXED ? sweep_split(handed, grid64, target64, nunits64).parts : 1;
    int32_t *cnt_out = &S.cnt[(k + 1) % 3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane & 7, slot = tid >> 3;
    for (int t = tid; t < nnz; t += kGroupBlock) {
        gidx[t] = (unsigned char)T.gidx[t];
        if (MIXED) reinterpret_cast<float *>(coef)[t] = T.gcoef32[t];
        else reinterpret_cast<double *>(coef)[t] = T.gcoef[t];
    }
    for (int t = tid; t <= npairs; t += kGroupBlock) gstart[t] = T.gstart[t];
    const bool reg = np.gamma != 0.0;
    for (int base = blockIdx.x * kGroupCells; base < cnt_in; base += gridDim.x * kGroupCells) {
        __syncthreads();  // the previous pass has read its shared memory
        if (tid < kGroupCells) {
            const int c = base + tid < cnt_in ? list_in[base + tid] : -1;
            scell[tid] = c;
            sh64[tid] = MIXED && c >= 0 ? S.h64[c] : 0;
        }
        __syncthreads();
        // this cell's state, on its way while the moments are loaded
        const int cell = scell[slot];
        const bool valid = cell >= 0, h32 = MIXED && !sh64[slot];
        const size_t off = (size_t)(valid ? cell : 0) * n;
        const int ph = valid ? S.phase[cell] : PH_DONE;
        const double lam = ph == PH_NEWTON ? S.lam[cell] : 0.0;
        double at[SL], ua[SL], gr[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int c = g + 8 * s;
            const bool in = valid && c < n;
            const double al = in ? S.alpha[off + c] : 0.0;
            at[s] = in && ph == PH_NEWTON ? fma(lam, S.dir[off + c], al) : al;
            ua[s] = in ? u[off + c] : 0.0;
            // for alpha.u below: component c of the pass's cells, rotated so that neither side conflicts
            if (c < n) {
                sH[c * kGroupCells + (slot ^ ((c & 7) << 2))] = at[s];
                sH[(n + c) * kGroupCells + (slot ^ ((c & 7) << 2))] = ua[s];
            }
        }
        double fs0 = 0.0, f0 = 0.0, gd0 = 0.0, gnorm0 = 0.0;  // of the accepted point (gnorm: squared)
        if (ph == PH_NEWTON) {
            fs0 = S.fsum[cell];
            f0 = S.f0[cell];
            gd0 = S.gd[cell];
            if (MIXED) gnorm0 = S.gnorm[cell];
        }
        const int ev = valid ? S.evals[cell] + 1 : 0;
        // the moments of the pass's cells, the sweeps' parts added in order: in FP32 for the
        // Hessian-only moments of tensor-core cells (accumulator values), else in FP64
        for (int e = tid; e < n2 * kGroupCells; e += kGroupBlock) {
            const int c = e / kGroupCells, j = e % kGroupCells;
            const int f = MIXED ? sh64[j] : 0;  // 1 + place among the handed cells
            const double *col = Vacc + (size_t)c * vs + min(base + j, cnt_in - 1);
            if (MIXED && c >= n && !sh64[j]) {
                float v = d2f_bits(col[0]);
#pragma unroll 4
                for (int p = 1; p < parts; ++p) v += d2f_bits(col[(size_t)p * cnt_in]);
                sVf[c * kGroupPitch + j] = v;
            } else {
                const int np_ = f ? parts64 : parts, step = f ? handed : cnt_in;
                const double *more = f ? Vacc + (size_t)c * vs + vs_handed + f - 1 : col + cnt_in;
                double v = col[0];
#pragma unroll 4
                for (int p = 1; p < np_; ++p) v += more[(size_t)(p - 1) * step];
                sV[c * kGroupPitch + j] = v;
                if (MIXED) sVf[c * kGroupPitch + j] = d2f_bits(v);
            }
        }
        __syncthreads();
        // alpha.u in the order of the components, as in the predictor and the thread-per-cell kernel: the
        // line search compares sums of terms far larger than themselves where alpha is large, and
        // summed over the lanes in a tree twice as many badly conditioned closures stalled in it. A
        // thread per cell, so that an FP64 instruction serves the block's 32 (in every group, by
        // shuffles, the M_3 mixed pass took 2.5% longer).
        if (tid < kGroupCells) {
            double sum = 0.0, sq = 0.0;
#pragma unroll
            for (int c = 0; c < n; ++c) {
                const double x = sH[c * kGroupCells + (tid ^ ((c & 7) << 2))];
                sum = fma(x, sH[(n + c) * kGroupCells + (tid ^ ((c & 7) << 2))], sum);
                if (reg && c >= np.reg0) sq = fma(x, x, sq);
            }
            sAu[tid] = sum;
            if (reg) sAu[kGroupCells + tid] = sq;
        }
        const double *V = sV + slot;
        const float *Vf = sVf + slot;
        bool fin = true;
        for (int c = g; c < n2; c += 8)
            fin = fin && (c < n || !h32 ? finite_bits(V[c * kGroupPitch])
                                        : (__float_as_uint(Vf[c * kGroupPitch]) & 0x7f800000u) != 0x7f800000u);
        const bool finite = ((~__ballot_sync(kFull, fin) >> (lane & 24)) & 0xffu) == 0;
        __syncthreads();
        const double au = sAu[slot], ar2 = reg ? sAu[kGroupCells + slot] : 0.0;
        const double fs = V[0] * T.rm0;
        const double ft = reg ? fma(0.5 * np.gamma, ar2, fs - au) : fs - au;
        bool accept = valid && finite;
        if (ph == PH_NEWTON) {
            const double slack = 64.0 * 2.220446049250313e-16 * (fs0 + fabs(fs0 - f0));
            accept = accept && ft <= f0 + np.c1 * lam * gd0 + slack;
        }
        // the Newton direction -H^-1 (<m e> - u + gamma alpha^r) of the accepted cells
        double y[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const int c = g + 8 * s;
            gr[s] = c < n ? V[c * kGroupPitch] - ua[s] : 0.0;
            if (reg && c < n && c >= np.reg0) gr[s] = fma(np.gamma, at[s], gr[s]);
            y[s] = 0.0;
        }
        const int reg0 = reg ? np.reg0 : n;
        bool spd = false;
        if (MIXED && __any_sync(kFull, accept && h32)) {
            float yf[SL];
#pragma unroll
            for (int s = 0; s < SL; ++s) yf[s] = -d2f_bits(gr[s]);
            float *Hs = reinterpret_cast<float *>(sH + warp * 4 * npairs) + (lane >> 3) * npairs;
            const bool ok = group_factor_solve<NN, float>(reinterpret_cast<const float *>(coef), gidx, gstart, Vf, Hs,
                                                          (float)np.gamma, reg0, g, yf);
            if (h32) {
                spd = ok;
#pragma unroll
                for (int s = 0; s < SL; ++s) y[s] = f2d_bits(yf[s]);
            }
            const unsigned keep = __ballot_sync(kFull, accept && h32 && ok);
            const float *W = reinterpret_cast<const float *>(sH + warp * 4 * npairs);
            for (int e = lane; e < 4 * npairs; e += 32) {
                const int q = e / npairs;
                if ((keep >> (8 * q)) & 1)
                    S.L[(size_t)scell[warp * 4 + q] * npairs + (e - q * npairs)] = f2d_bits(W[e]);
            }
            __syncwarp();
        }
        if (!MIXED || __any_sync(kFull, accept && !h32)) {
            double yd[SL];
#pragma unroll
            for (int s = 0; s < SL; ++s) yd[s] = -gr[s];
            double *Hs = sH + slot * npairs;
            bool ok;
            if constexpr (MIXED)
                ok = group_factor_solve_shared<NN>(T, V, Hs, np.gamma, reg0, g, yd);
            else
                ok = group_factor_solve<NN, double>(reinterpret_cast<const double *>(coef), gidx, gstart, V, Hs,
                                                    np.gamma, reg0, g, yd);
            if (!h32) {
                spd = ok;
#pragma unroll
                for (int s = 0; s < SL; ++s) y[s] = yd[s];
            }
            const unsigned keep = __ballot_sync(kFull, accept && !h32 && ok);
            const double *W = sH + warp * 4 * npairs;
            for (int e = lane; e < 4 * npairs; e += 32) {
                const int q = e / npairs;
                if ((keep >> (8 * q)) & 1) S.L[(size_t)scell[warp * 4 + q] * npairs + (e - q * npairs)] = W[e];
            }
            __syncwarp();
        }
        double gn2 = 0.0, un2 = 0.0, gd = 0.0;
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            gn2 = fma(gr[s], gr[s], gn2);
            un2 = fma(ua[s], ua[s], un2);
            gd = fma(gr[s], y[s], gd);
        }
        gn2 = group_sum(gn2);
        un2 = group_sum(un2);
        gd = group_sum(gd);
        const bool step = accept && spd;
        if (step) {
#pragma unroll
            for (int s = 0; s < SL; ++s) {
                const int c = g + 8 * s;
                if (c < n) {
                    S.alpha[off + c] = at[s];
                    S.U[off + c] = V[c * kGroupPitch];
                    S.dir[off + c] = y[s];
                }
            }
        }
        bool cont = false;
        if (g == 0 && valid) {
            S.evals[cell] = ev;
            int code = 0;  // status of a cell that fails here
            if (step) {
                S.fsum[cell] = fs;
                S.f0[cell] = ft;
                if (S.lfac) S.lfac[cell] = 1;
                int iters = S.iters[cell];
                if (ph == PH_NEWTON) ++iters;
                S.iters[cell] = iters;
                if (gn2 <= np.tau * np.tau * un2) {
                    S.phase[cell] = PH_DONE;
                } else if (iters >= np.max_iter) {
                    code = KITRT_ENOCONVERGE;
                } else {
                    // a Newton step on the tensor-core Hessian that does not halve the residual
                    // sends the cell to the FP64 Hessian
                    if (MIXED && ph == PH_NEWTON && gn2 > kStallRatio * kStallRatio * gnorm0) hand_over(S, cell);
                    if (MIXED) S.gnorm[cell] = gn2;
                    S.gd[cell] = gd;
                    S.lam[cell] = 1.0;
                    S.halv[cell] = 0;
                    S.phase[cell] = PH_NEWTON;
                    cont = true;
                }
            } else if (accept) {
                // FP32 rounding broke positive definiteness: redo this point with the FP64 Hessian;
                // no further fallback there
                if (h32) {
                    hand_over(S, cell);
                    cont = true;
                } else {
                    code = KITRT_ECHOL;
                }
            } else if (ph == PH_INIT) {
                code = KITRT_ENOTREALIZABLE;
            } else {
                const int h = S.halv[cell] + 1;
                if (h <= np.max_halvings) {
                    S.halv[cell] = h;
                    S.lam[cell] = 0.5 * lam;
                    cont = true;
                } else if (h32) {
                    // the line search could not follow the direction from the tensor-core Hessian:
                    // restart from the accepted point with the FP64 Hessian
                    hand_over(S, cell);
                    S.halv[cell] = 0;
                    S.phase[cell] = PH_INIT;
                    cont = true;
                } else {
                    code = KITRT_ELINESEARCH;
                }
            }
            if (code) {
                S.status[cell] = code;
                S.phase[cell] = PH_DONE;
                atomicAdd(&S.cnt[3], 1);
            }
        }
        __syncwarp();
        // every listed cell of this pass is one evaluation
        const unsigned live = __ballot_sync(kFull, valid && g == 0);
        const int evmax = __reduce_max_sync(kFull, ev);
        if (lane == 0 && live) {
            atomicAdd(&S.cnt[6], __popc(live));
            atomicMax(&S.cnt[4], evmax);
        }
        const int at_out = push_agg(list_out, cnt_out, cell, cont);
        if (MIXED && cont && S.h64[cell]) {
            const int f = atomicAdd(&S.cnt[12 + (k + 1) % 3], 1);
            S.handed[(k + 1) & 1][f] = at_out;
            S.h64[cell] = 1 + f;
        }
    }
}

}  // namespace kitrt_dev
