// FP64 entropy closure: Newton's method on the dual of the minimum-entropy problem
// [Sec. 3.1, Eq. entropyOCP; Maxwell-Boltzmann entropy], with Armijo backtracking.
//
// A round evaluates every listed cell at its trial point and takes its Newton step, in two kernels:
//  - the sweep (a thread per cell and part of the quadrature) forms the degree-2N moments
//      V_c = sum_q w_q exp(alpha.m_q) m~_c(q)
//    in the sum-factorised fixed-point form of sweep.cuh, so that U = V[0:n] are the ansatz moments,
//    <exp(alpha.m)> = V_0 / m_0 and the Hessian H_ab = sum_c G_abc V_c (Gaunt coefficients) comes
//    without per-point pair products;
//  - the Newton kernel (newton_common.cuh: 8 lanes or a thread per cell) adds the parts, decides the line
//    search, factorises the Hessian and finds the next direction.
// Here are also the start of a closure (continuation test, predictor), its end (alpha, FP64 ansatz) and the
// allocation-free closure's kernel, a warp per cell in FP64.
//
// Cells that still iterate are kept in a compacted list; every round advances each listed cell by one
// evaluation (one trial point of the line search) and writes the cells that continue into the next
// list. Counters rotate over three slots so that no launch has to clear the slot it fills.
#include <math.h>

#include "async_copy.cuh"
#include "kitrt_internal.cuh"
#include "kexp.cuh"
#include "newton_common.cuh"
#include "sweep.cuh"

namespace {

using namespace kitrt_dev;
constexpr int kWarps = 8;  // warps per block
constexpr int kThreadBlock = 64;  // block of the thread-per-cell Newton kernels

// ---------------------------------------------------------------------------------------------
// begin: start a closure. first == 1: every cell starts from alpha_in with an evaluation.
// first == 0: the previous closure left alpha_k, its moments U, <exp>, and the Cholesky factor
// of H(alpha_k); with the new u the gradient is U - u. One thread per cell tests it: a cell
// already converged (and with no polish step to take) is done at once; the others go to the
// predictor list, where predict_kernel takes the first Newton direction from the stored factor
// without a new quadrature pass.
// first == 2: per cell, the second case when alpha_in is bit for bit the alpha the last closure
// returned for this cell (alpha_k, plus the polish step when polishing) and that closure
// succeeded, so the stored state is exactly the state behind the given alpha; the first case
// otherwise (the cell's stored <exp> is then poisoned, so that the learned pass cannot mistake
// it for a previous point).
// renew: a converged cell is evaluated all the same, so that the sweeps write its ansatz (the closure
// that left its state wrote none).
// ---------------------------------------------------------------------------------------------

// Warp-aggregated append of `cell` to a list when pred holds (all active lanes call it).
__device__ __forceinline__ void push_if(int32_t *list, int32_t *cnt, int cell, bool pred)
{
    const unsigned act = __activemask();
    const unsigned m = __ballot_sync(act, pred);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(act, base, leader);
    if (pred) list[base + __popc(m & ((1u << lane) - 1u))] = cell;
}

template <int NN>
__global__ void __launch_bounds__(256)
begin_test_kernel(NewtonState S, const double *__restrict__ u, const double *__restrict__ alpha_in,
                  int first, NewtonParams np, int C, int learned, int renew)
{
    constexpr int n = Dims<NN>::n;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < C; cell += gridDim.x * blockDim.x) {
        const size_t off = (size_t)cell * n;
        bool cold = first == 1;
        if (first == 2) {
            // the alpha the finish kernel returned: alpha_k (+ the polish step when polishing)
            bool same = S.status[cell] == 0;
#pragma unroll
            for (int a = 0; a < n; ++a) {
                double out = S.alpha[off + a];
                if (np.polish) out += S.dir[off + a];
                same = same && __double_as_longlong(out) == __double_as_longlong(alpha_in[off + a]);
            }
            cold = !same;
        }
        S.iters[cell] = 0;
        S.halv[cell] = 0;
        S.evals[cell] = 0;
        S.status[cell] = 0;
        if (S.h64) S.h64[cell] = 0;
        if (S.gnorm) S.gnorm[cell] = INFINITY;
        bool to_eval = false, to_predict = false;
        if (cold) {
#pragma unroll
            for (int a = 0; a < n; ++a) S.alpha[off + a] = alpha_in[off + a];
            S.phase[cell] = PH_INIT;
            if (first == 2) S.fsum[cell] = __longlong_as_double(0x7ff8000000000000LL);
            // learned closures go to the network first (the predictor list doubles as its list)
            to_eval = !learned;
            to_predict = learned;
        } else {
            double gn2 = 0.0, un2 = 0.0;
#pragma unroll
            for (int a = 0; a < n; ++a) {
                const double ua = u[off + a];
                double g = S.U[off + a] - ua;
                if (a >= np.reg0) g = fma(np.gamma, S.alpha[off + a], g);
                gn2 = fma(g, g, gn2);
                un2 = fma(ua, ua, un2);
            }
            if (gn2 <= kRoundoff2 * un2 || (!np.polish && gn2 <= np.tau * np.tau * un2)) {
                // already converged and no polish step to take (the polish is off, or the residual
                // is at round-off, where it would move alpha by less than its own rounding)
#pragma unroll
                for (int a = 0; a < n; ++a) S.dir[off + a] = 0.0;
                S.phase[cell] = renew ? PH_INIT : PH_DONE;
                to_eval = renew;
            } else {
                to_predict = true;
            }
        }
        push_if(S.list[0], &S.cnt[0], cell, to_eval);
        push_if(S.list[1], &S.cnt[8], cell, to_predict);
    }
}

// One thread per listed cell: every FP64 instruction of the triangular solves keeps all 32 lanes
// busy, and one warp per scheduler already fills the FP64 pipe (64 cycles per instruction). For
// N <= 3 the factor is read into registers. For N >= 4 (120 or 231 entries) a block of one warp
// copies its 32 cells' factors into shared memory (asynchronously, whole rows at a time: read by the
// threads themselves each load touches 32 lines) and works from there, the vector in shared memory
// too. M_5, 996,872 cells: a warp per cell took 8.2 ms a step, strided reads 7.0, whole factors in
// shared memory (3 warps on an SM) 3.4, with the test that precedes it. SEG (M_5, more cells than those 3
// warps on every SM take at once) stages the rows in segments of at most kSegPairs entries, each but
// the last once more for the backward solve, so that 8 warps fit: 2.2 ms. For M_4 whole factors leave
// room for 6 warps, and segments gain nothing: the test and two predictors on 20,000, 178,802 and
// 498,002 cells take 0.092, 0.511 and 1.320 ms whole, 0.093, 0.537 and 1.326 in segments.
template <int NN, bool SEG>
struct PredictDims {
    static constexpr bool in_regs = NN <= 3;
    static constexpr int threads = in_regs ? kThreadBlock : 32;
    static constexpr int kSegPairs = SEG ? 79 : Dims<NN>::npairs;
    static constexpr int pitch = kSegPairs | 1;  // odd: a column of 32 rows is free of conflicts
    // end of the segment of rows that starts at row r
    static __host__ __device__ constexpr int seg_end(int r)
    {
        int e = r;
        while (e < Dims<NN>::n && (e + 1) * (e + 2) / 2 - r * (r + 1) / 2 <= kSegPairs) ++e;
        return e;
    }
    static constexpr size_t smem = in_regs ? 0 : sizeof(double) * 32 * (pitch + Dims<NN>::n);
};

template <int NN, bool SEG>
__global__ void __launch_bounds__(PredictDims<NN, SEG>::threads)
predict_kernel(NewtonState S, const double *__restrict__ u, NewtonParams np, const int32_t *__restrict__ list,
               const int32_t *__restrict__ count)
{
    using D = PredictDims<NN, SEG>;
    constexpr int n = Dims<NN>::n, npairs = Dims<NN>::npairs;
    extern __shared__ __align__(16) double predict_smem[];  // [32][pitch] factors, [n][32] vectors
    const int cnt = *count;
    const int stride = gridDim.x * blockDim.x;
    const int rounds = (cnt + stride - 1) / stride;
    for (int rd = 0; rd < rounds; ++rd) {
        const int it = rd * stride + blockIdx.x * blockDim.x + threadIdx.x;
        bool cont = false;
        int cell = it < cnt ? list[it] : -1;
        // rows [r0, r1) of the warp's factors into shared memory
        auto stage = [&](int r0, int r1) {
            const int p0 = tri_idx(r0, 0), len = tri_idx(r1, 0) - p0;
            __syncwarp();
            for (int r = 0; r < 32; ++r) {
                const int c = __shfl_sync(kFull, cell, r);
                if (c < 0) break;
                const double *row = S.L + (size_t)c * npairs + p0;
                for (int p = threadIdx.x; p < len; p += 32) kitrt_async::cp_async8(predict_smem + r * D::pitch + p, row + p);
            }
            kitrt_async::cp_async_wait_all();
            __syncwarp();
        };
        // with segments every lane of the warp takes part in the staging
        if (!D::in_regs || it < cnt) {
            const bool mine = it < cnt;
            const size_t off = (size_t)(mine ? cell : 0) * n;
            double gn2 = 0.0, un2 = 0.0, au = 0.0, ar2 = 0.0, gd = 0.0;
            auto gradient = [&](int a) {
                const double ua = u[off + a], al = S.alpha[off + a];
                double g = S.U[off + a] - ua;
                if (a >= np.reg0) {
                    g = fma(np.gamma, al, g);
                    ar2 = fma(al, al, ar2);
                }
                gn2 = fma(g, g, gn2);
                un2 = fma(ua, ua, un2);
                au = fma(al, ua, au);
                return g;
            };
            // d = -H^-1 g with the stored factor (1/L_jj on its diagonal)
            if constexpr (D::in_regs) {
                const double *L = S.L + (size_t)cell * npairs;
                double Lp[npairs], y[n], g[n];
#pragma unroll
                for (int p = 0; p < npairs; ++p) Lp[p] = L[p];
#pragma unroll
                for (int a = 0; a < n; ++a) {
                    g[a] = gradient(a);
                    y[a] = -g[a];
                }
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    double t = y[i];
#pragma unroll
                    for (int k = 0; k < i; ++k) t = fma(-Lp[tri_idx(i, k)], y[k], t);
                    y[i] = t * Lp[tri_idx(i, i)];
                }
#pragma unroll
                for (int i = n - 1; i >= 0; --i) {
                    double t = y[i];
#pragma unroll
                    for (int k = i + 1; k < n; ++k) t = fma(-Lp[tri_idx(k, i)], y[k], t);
                    y[i] = t * Lp[tri_idx(i, i)];
                }
#pragma unroll
                for (int a = 0; a < n; ++a) {
                    S.dir[off + a] = y[a];
                    gd = fma(g[a], y[a], gd);
                }
            } else {
                const double *L = predict_smem + threadIdx.x * D::pitch;
                double *y = predict_smem + 32 * D::pitch + threadIdx.x;
                int r0 = 0;
#pragma unroll 1
                for (int r1 = D::seg_end(0);; r0 = r1, r1 = D::seg_end(r1)) {
                    stage(r0, r1);
                    if (mine) {
#pragma unroll 1
                        for (int i = r0; i < r1; ++i) {
                            const double *row = L + tri_idx(i, 0) - tri_idx(r0, 0);
                            double t = -gradient(i);
#pragma unroll 4
                            for (int k = 0; k < i; ++k) t = fma(-row[k], y[k * 32], t);
                            t *= row[i];
                            y[i * 32] = t;
                            gd = fma(-t, t, gd);  // g . d = -|L^-1 g|^2
                        }
                    }
                    if (r1 == n) break;
                }
                // backward from the last segment, which is still there
#pragma unroll 1
                for (int r1 = n;;) {
                    if (mine) {
#pragma unroll 1
                        for (int i = r1 - 1; i >= r0; --i) {
                            const double *row = L + tri_idx(i, 0) - tri_idx(r0, 0);
                            const double x = y[i * 32] * row[i];
                            S.dir[off + i] = x;
#pragma unroll 4
                            for (int k = 0; k < i; ++k) y[k * 32] = fma(-row[k], x, y[k * 32]);
                        }
                    }
                    if (r0 == 0) break;
                    r1 = r0;
                    for (r0 = 0; D::seg_end(r0) < r1;) r0 = D::seg_end(r0);
                    stage(r0, r1);
                }
            }
            if (!mine) {
                // a lane without a cell
            } else if (gn2 <= np.tau * np.tau * un2) {
                S.phase[cell] = PH_DONE;  // converged; d is the polish step
            } else {
                if (S.gnorm) S.gnorm[cell] = gn2;
                S.f0[cell] = fma(0.5 * np.gamma, ar2, S.fsum[cell] - au);
                S.gd[cell] = gd;
                S.lam[cell] = 1.0;
                S.phase[cell] = PH_NEWTON;
                cont = true;
            }
        }
        push_agg(S.list[0], &S.cnt[0], cell, cont);
    }
}

// ---------------------------------------------------------------------------------------------
// eval: one trial point per listed cell (alpha + lam dir, or alpha itself for PH_INIT), then the
// Armijo decision, and on acceptance the Hessian, its Cholesky factor, the convergence test and
// the next Newton direction.
// ---------------------------------------------------------------------------------------------
// One warp per listed cell, sums and Newton logic in one kernel without an accumulator: the
// allocation-free closure.
template <int NN>
__global__ void __launch_bounds__(kWarps * 32)
eval_kernel(Tables T, NewtonState S, const double *__restrict__ u, int k, NewtonParams np)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2;
    __shared__ double sH[kWarps][n * n];
    __shared__ double sV[kWarps][n2];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int32_t *list_in = S.list[k & 1];
    int32_t *list_out = S.list[(k + 1) & 1];
    const int cnt_in = S.cnt[k % 3];
    int32_t *cnt_out = &S.cnt[(k + 1) % 3];
    if (blockIdx.x == 0 && threadIdx.x == 0) S.cnt[(k + 2) % 3] = 0;
    double *H = sH[wib];
    double *Vs = sV[wib];
    const int Qp = T.Qp;
    const double *__restrict__ Mt = T.Mt;
    const double *__restrict__ wq = T.w;
    for (int it = blockIdx.x * kWarps + wib; it < cnt_in; it += gridDim.x * kWarps) {
        const int cell = list_in[it];
        const size_t off = (size_t)cell * n;
        const int ph = S.phase[cell];
        const double ua = lane < n ? u[off + lane] : 0.0;
        const double al = lane < n ? S.alpha[off + lane] : 0.0;
        const double lam = ph == PH_NEWTON ? S.lam[cell] : 0.0;
        const double di = (ph == PH_NEWTON && lane < n) ? S.dir[off + lane] : 0.0;
        const double at = lane < n ? fma(lam, di, al) : 0.0;
        double atv[n];
#pragma unroll
        for (int a = 0; a < n; ++a) atv[a] = __shfl_sync(kFull, at, a);

        double V[n2];
#pragma unroll
        for (int c = 0; c < n2; ++c) V[c] = 0.0;
        for (int q = lane; q < Qp; q += 32) {
            double z = 0.0;
#pragma unroll
            for (int a = 0; a < n; ++a) z = fma(atv[a], Mt[a * Qp + q], z);
            const double e = wq[q] * kexp(z, T.exptab);
#pragma unroll
            for (int c = 0; c < n2; ++c) V[c] = fma(e, Mt[c * Qp + q], V[c]);
        }
#pragma unroll
        for (int c = 0; c < n2; ++c) V[c] = warp_sum(V[c]);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < n2; ++c)
            if (lane == (c & 31)) Vs[c] = V[c];
        __syncwarp();
        newton_post<NN>(T, S, np, cell, ph, lam, at, ua, Vs, H, list_out, cnt_out, lane);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------------
// Sweep of the FP64 mode: one thread per listed cell (tiles of 128), every degree-2N moment in the
// sum-factorised fixed-point form of sweep.cuh. Work items are (tile, part of the quadrature); each
// stores its partial moments with plain stores into its own column block of Vacc, which the
// Newton kernel adds in order, so the result does not depend on scheduling.
// ---------------------------------------------------------------------------------------------
constexpr int kSweepThreads = 128;
// Quads per unit of the split of these sweeps: half of the tensor-core sweep's chunk, so that small
// lists spread over more SMs (M_2, 3,872 cells: 0.16 -> 0.135 ms in two steps; handed-over cells of a
// checkerboard, 25,088 cells, four closures: 0.24 -> 0.21 ms).
constexpr int kUnit64 = 4;
int units64(int nquad) { return (nquad + kUnit64 - 1) / kUnit64; }

// An exponential of the sweeps as a double, with the range test that fx_double leaves out (rows outside the
// fixed-point range reach 2^-1024).
__device__ __forceinline__ double fx_psi(const Exp &e) { return e.m < -1022 ? 0.0 : kitrt_fx::fx_double(e); }

// Dynamic shared memory of sweep64_kernel: the exp table, the moments [n2][thread] and the trial
// alpha's limbs [n][thread], the azimuthal factors.
size_t sweep64_smem(int n, int n2, int N, int J)
{
    return 2048 * 8 + (size_t)(n2 + n) * kSweepThreads * 8 + (size_t)J * 4 * N * 8;
}

// Which cells a sweep takes, and what it writes besides the moments.
enum class Cells {
    kListed,   // FP64 mode: the listed cells at their trial points
    kHanded,   // mixed modes: the cells handed over to the FP64 Hessian (positions in the list), their
               // trial points' FP32 ansatz into psi; the first part goes to the cell's own column, the
               // others to columns from C on
    kGiven     // every cell at the given alpha (one part), its FP64 ansatz into psi (the adjoint)
};

template <int NN, Cells CELLS>
__global__ void __launch_bounds__(kSweepThreads)
sweep64_kernel(Tables T, NewtonState S, const double *__restrict__ u, int k, double *__restrict__ Vacc, int vs,
               int target_items, const double *__restrict__ alpha, void *__restrict__ psi, int C)
{
    constexpr bool GIVEN = CELLS == Cells::kGiven, HANDED = CELLS == Cells::kHanded;
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2, L2 = 2 * NN;
    extern __shared__ __align__(16) unsigned char sweep_smem[];
    uint64_t *tab = (uint64_t *)sweep_smem;
    long long *sV = (long long *)(tab + 2048);
    int2 *sA = (int2 *)(sV + n2 * kSweepThreads);
    int2 *trig = sA + n * kSweepThreads;
    const int32_t *list_in = GIVEN ? nullptr : S.list[k & 1];
    const int32_t *pos_in = HANDED ? S.handed[k & 1] : nullptr;
    const int cnt_in = GIVEN ? C : HANDED ? S.cnt[12 + k % 3] : S.cnt[k % 3];
    if (HANDED && cnt_in == 0) return;
    if (CELLS == Cells::kListed && blockIdx.x == 0 && threadIdx.x == 0) S.cnt[(k + 2) % 3] = 0;
    const int nunits = (T.nquad + kUnit64 - 1) / kUnit64;
    const SweepSplit sp = sweep_split(cnt_in, gridDim.x, GIVEN ? 0 : target_items, nunits);
    const int items = sp.tiles * sp.parts;
    if ((int)blockIdx.x >= items) return;
    for (int j = threadIdx.x; j < 2048; j += kSweepThreads) tab[j] = T.fx_exp[j];
    for (int j = threadIdx.x; j < T.J * 2 * L2; j += kSweepThreads) trig[j] = T.fx_trig[j];
    __syncthreads();
    long long *mine = sV + threadIdx.x;
    int2 *myA = sA + threadIdx.x;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int tile = item / sp.parts, part = item % sp.parts;
        const int slot = tile * kSweepThreads + threadIdx.x;
        if (slot >= cnt_in) continue;  // threads are independent: no block barrier below
        const int q_begin = part * nunits / sp.parts * kUnit64;
        const int q_end = min(T.nquad, (part + 1) * nunits / sp.parts * kUnit64);
        const int cell = GIVEN ? slot : list_in[HANDED ? pos_in[slot] : slot];
        const double *al = (GIVEN ? alpha : S.alpha) + (size_t)cell * n, *di = GIVEN ? al : S.dir + (size_t)cell * n;
        const double lam = !GIVEN && S.phase[cell] == PH_NEWTON ? S.lam[cell] : 0.0;
        float bound = 0.0f;
#pragma unroll
        for (int a = 0; a < n; ++a) {
            const double x = lam != 0.0 ? fma(lam, di[a], al[a]) : al[a];
            const Limb w = kitrt_fx::split<32>(kitrt_fx::fx_from_double(x));
            myA[a * kSweepThreads] = make_int2(w.h, w.l);
            bound = fmaf(fabsf(d2f_bits(x)), T.fx_mmax[a], bound);
        }
        // rows outside the range are scaled down; beyond that (-1) they take FP64 exponentials
        const int sh = fx_row_shift(bound);
        if (sh > 0) fx_scale_limbs(al, di, lam, 0, 1, n, sh, myA, kSweepThreads);
        bool bad = false;
#pragma unroll
        for (int c = 0; c < n2; ++c) mine[c * kSweepThreads] = 0;
        long long A0 = 0;
        Limb A[2 * NN];
        FxSums<L2> B;
        B.clear();
        B.Sx = kitrt_fx::fx_scale_of(u[(size_t)cell * n]);
        auto trial = [&](int a) {
            const int2 v = myA[a * kSweepThreads];
            return Limb{v.x, v.y};
        };
        auto moment = [&](int c) -> long long & { return mine[c * kSweepThreads]; };
        int ring = q_begin / T.J, jq = q_begin - ring * T.J;
        bool fresh = true;
#pragma unroll 1
        for (int qd = q_begin; qd < q_end; ++qd) {
            if (fresh) {
                fx_coeffs<NN>(trial, T.fx_ringA + (size_t)ring * n, A0, A);
                fresh = false;
            }
            const int2 *tr = trig + jq * 2 * L2;
            const int pa = quad_pair0(ring, jq, T.P), pb = quad_pair1(ring, jq, T.P);
            Exp e[4];
            long long s[4];
            fx_exponents<NN>(A0, A, tr, L2, jq == 0, s);
            if (sh != 0)
                bad = !fx_outside_quad<NN>(sh, T, point_of(S, GIVEN ? alpha : nullptr),
                                           GIVEN ? slot : list_in[HANDED ? pos_in[slot] : slot], pa, pb, s) || bad;
#pragma unroll
            for (int t = 0; t < 4; ++t) e[t] = kitrt_fx::fx_exp(s[t], tab);
            if (HANDED) {
                // ansatz of the trial point (the last accepted trial leaves the solution's)
                if (psi) {
                    float *row = (float *)psi + (size_t)cell * T.Qp;
                    float f[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) f[t] = __uint_as_float(kitrt_fx::fx_float_bits(e[t]));
                    *(float2 *)(row + 2 * pa) = make_float2(f[0], f[1]);
                    if (pb >= 0) *(float2 *)(row + 2 * pb) = make_float2(f[2], f[3]);
                }
            }
            if (GIVEN) {
                double *row = (double *)psi + (size_t)cell * T.Qp;
                *(double2 *)(row + 2 * pa) = make_double2(fx_psi(e[0]), fx_psi(e[1]));
                if (pb >= 0) *(double2 *)(row + 2 * pb) = make_double2(fx_psi(e[2]), fx_psi(e[3]));
            }
            if (pb < 0) e[2] = e[3] = Exp{0, -100000};
            fx_accumulate<L2>(e, tr, L2, jq == 0, qd == q_begin, B, [&](int d) {
                for (int c = 0; c < n2; ++c) mine[c * kSweepThreads] = kitrt_fx::sar(mine[c * kSweepThreads], d);
            });
            if (++jq == T.J) {
                fx_flush<L2>(T.fx_ringW + (size_t)ring * n2, T.fx_sumshift, B, moment);
                jq = 0;
                ++ring;
                fresh = true;
            }
        }
        if (!fresh) fx_flush<L2>(T.fx_ringW + (size_t)ring * n2, T.fx_sumshift, B, moment);
        double *col = Vacc + (!HANDED ? (size_t)part * cnt_in + slot
                              : part ? (size_t)C + (size_t)(part - 1) * cnt_in + slot : (size_t)pos_in[slot]);
        const int unit = fx_unit(B.Sx, T);
#pragma unroll 4
        for (int c = 0; c < n2; ++c)
            col[(size_t)c * vs] = bad ? __longlong_as_double(0x7ff8000000000000LL)
                                      : kitrt_fx::fx_to_double(mine[c * kSweepThreads], unit);
    }
}

// ---------------------------------------------------------------------------------------------
// finish: final alpha (alpha_k plus the polish step if enabled) to the caller and the FP64 ansatz psi
// at every folded point. Lanes are cells; the block's 4 warps take a quarter of the quads each of the
// same 32 cells, in the fixed-point form of the sweeps (exponents of four azimuths from one set of
// products). FP64 exponents and exponentials (18 FP64 instructions a point for M_3) bound the former
// kernel (a warp per cell): 1.23 -> 0.33 ms a step on 99,458 cells, M_3, order 20, where 318 MB are
// written.
// ---------------------------------------------------------------------------------------------
constexpr int kFinishWarps = 4;

template <int NN>
__device__ __noinline__ void psi_row_fp64(const Tables &T, const double *alpha, double *row, int q0, int q1)
{
    constexpr int n = Dims<NN>::n;
    for (int q = q0; q < q1; ++q) {
        double z = 0.0;
        for (int b = 0; b < n; ++b) z = fma(alpha[b], T.Mt[(size_t)b * T.Qp + q], z);
        row[q] = kexp(z, T.exptab);
    }
}

template <int NN>
__global__ void __launch_bounds__(kFinishWarps * 32)
finish_kernel(Tables T, NewtonState S, double *__restrict__ alpha_out, double *__restrict__ psi, int polish,
              int compare_prev, int C)
{
    constexpr int n = Dims<NN>::n;
    extern __shared__ __align__(16) unsigned char finish_smem[];
    uint64_t *tab = (uint64_t *)finish_smem;
    int2 *trig = (int2 *)(tab + 2048);                 // [J][2 NN]
    int2 *sA = trig + T.J * 2 * NN;                    // [n][32]
    float *sB = (float *)(sA + n * 32);                // [warp][32]
    int *sDiff = (int *)(sB + kFinishWarps * 32);      // [warp][32]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if ((int)blockIdx.x * 32 >= C) return;
    for (int e = tid; e < 2048; e += blockDim.x) tab[e] = T.fx_exp[e];
    for (int e = tid; e < T.J * 2 * NN; e += blockDim.x) {
        const int p = e / (2 * NN), q = e % (2 * NN);
        trig[e] = T.fx_trig[p * 4 * NN + (q < NN ? q : NN + q)];
    }
    for (int base = blockIdx.x * 32; base < C; base += gridDim.x * 32) {
        const int cell = min(base + lane, C - 1);
        const size_t off = (size_t)cell * n;
        const bool add = polish && S.status[cell] == 0;
        __syncthreads();  // the tables, and the previous pass's reads of sA
        // every warp forms its share of the components; alpha_out still holds the previous step's
        // alpha (and psi its ansatz) when compare_prev is set: a bitwise-unchanged alpha leaves psi
        // as it is
        float bound = 0.0f;
        int differs = compare_prev ? 0 : 1;
        for (int c = warp; c < n; c += kFinishWarps) {
            double a = S.alpha[off + c];
            if (add) a += S.dir[off + c];
            if (compare_prev && !(alpha_out[off + c] == a)) differs = 1;
            const Limb w = kitrt_fx::split<32>(kitrt_fx::fx_from_double(a));
            sA[c * 32 + lane] = make_int2(w.h, w.l);
            bound = fmaf(fabsf(d2f_bits(a)), T.fx_mmax[c], bound);
            if (base + lane < C) alpha_out[off + c] = a;  // this thread alone reads and writes it
        }
        sB[tid] = bound;
        sDiff[tid] = differs;
        // a row outside the range has a quarter of the components outside a quarter of it
        const bool any_wide = __syncthreads_or(!(bound < kitrt_fx::kFxMaxZ / kFinishWarps));
        differs = 0;
        bound = 0.0f;
#pragma unroll
        for (int w = 0; w < kFinishWarps; ++w) {
            differs |= sDiff[w * 32 + lane];
            bound += sB[w * 32 + lane];
        }
        const int sh = fx_row_shift(bound);  // outside the range: scaled down; beyond that (-1) in FP64
        if (any_wide) {
            if (sh > 0)
                for (int c = warp; c < n; c += kFinishWarps) {
                    double a = S.alpha[off + c];
                    if (add) a += S.dir[off + c];
                    const Limb w = kitrt_fx::split<32>(kitrt_fx::fx_from_double(a, sh));
                    sA[c * 32 + lane] = make_int2(w.h, w.l);
                }
            __syncthreads();
        }
        const bool store = differs && base + lane < C;
        if (!__any_sync(kFull, store)) continue;
        const int qd0 = warp * T.nquad / kFinishWarps, qd1 = (warp + 1) * T.nquad / kFinishWarps;
        double *row = psi + (size_t)cell * T.Qp;
        if (store && sh < 0)
            psi_row_fp64<NN>(T, alpha_out + off, row, warp * T.Qf / kFinishWarps, (warp + 1) * T.Qf / kFinishWarps);
        int ring = qd0 / T.J, jq = qd0 - ring * T.J;
        bool fresh = true;
        long long A0 = 0;
        Limb A[2 * NN];
#pragma unroll 1
        for (int qd = qd0; qd < qd1; ++qd) {
            if (fresh) {
                fx_coeffs<NN>(
                    [&](int c) {
                        const int2 v = sA[c * 32 + lane];
                        return Limb{v.x, v.y};
                    },
                    T.fx_ringA + (size_t)ring * n, A0, A);
                fresh = false;
            }
            const int pa = quad_pair0(ring, jq, T.P), pb = quad_pair1(ring, jq, T.P);
            long long s[4];
            fx_exponents<NN>(A0, A, trig + jq * 2 * NN, NN, jq == 0, s);
            double e[4];
            if (sh == 0) {
#pragma unroll
                for (int t = 0; t < 4; ++t) e[t] = kitrt_fx::fx_double(kitrt_fx::fx_exp(s[t], tab));
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const bool ok = sh < 0 || kitrt_fx::fx_unscale(s[t], sh);
                    e[t] = ok ? fx_psi(kitrt_fx::fx_exp(s[t], tab)) : __longlong_as_double(0x7ff0000000000000LL);
                }
            }
            if (store && sh >= 0) {
                *(double2 *)(row + 2 * pa) = make_double2(e[0], e[1]);
                if (pb >= 0) *(double2 *)(row + 2 * pb) = make_double2(e[2], e[3]);
            }
            if (++jq == T.J) {
                jq = 0;
                ++ring;
                fresh = true;
            }
        }
    }
}

// finish without an ansatz to write (the mixed modes' sweeps already wrote it): the final alpha,
// element-wise over the C x n entries (coalesced, every lane busy).
__global__ void finish_alpha_kernel(NewtonState S, double *__restrict__ alpha_out, int polish, int n,
                                    int C)
{
    const size_t total = (size_t)C * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int cell = (int)(e / n);
        double a = S.alpha[e];
        if (polish && S.status[cell] == 0) a += S.dir[e];
        alpha_out[e] = a;
    }
}

// Degree-2N moments V_c = sum_q w_q exp(alpha.m_q) m~_c(q) of given alphas, in FP64.
template <int NN>
__global__ void __launch_bounds__(kWarps * 32)
moments_kernel(Tables T, const double *__restrict__ alpha, double *__restrict__ V, int C)
{
    constexpr int n = Dims<NN>::n, n2 = Dims<NN>::n2;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int Qp = T.Qp;
    for (int cell = blockIdx.x * kWarps + wib; cell < C; cell += gridDim.x * kWarps) {
        double av[n], acc[n2];
#pragma unroll
        for (int a = 0; a < n; ++a) av[a] = alpha[(size_t)cell * n + a];
#pragma unroll
        for (int c = 0; c < n2; ++c) acc[c] = 0.0;
        for (int q = lane; q < Qp; q += 32) {
            double z = 0.0;
#pragma unroll
            for (int a = 0; a < n; ++a) z = fma(av[a], T.Mt[a * Qp + q], z);
            const double e = T.w[q] * kexp(z, T.exptab);
#pragma unroll
            for (int c = 0; c < n2; ++c) acc[c] = fma(e, T.Mt[c * Qp + q], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < n2; ++c) {
            const double v = warp_sum(acc[c]);
            if (lane == 0) V[(size_t)cell * n2 + c] = v;
        }
    }
}

// Full Hessian H_ab = sum_c G_abc V_c (row-major n x n per cell) from degree-2N moments.
__global__ void gaunt_kernel(Tables T, const double *__restrict__ V, double *__restrict__ H, int C)
{
    const int n = T.n, n2 = T.n2, npairs = n * (n + 1) / 2;
    const size_t total = (size_t)C * npairs;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int cell = (int)(i / npairs), p = (int)(i % npairs);
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= p) ++a;
        const int b = p - a * (a + 1) / 2;
        double h = 0.0;
        for (int t = T.gstart[p]; t < T.gstart[p + 1]; ++t) h = fma(T.gcoef[t], V[(size_t)cell * n2 + T.gidx[t]], h);
        H[(size_t)cell * n * n + a * n + b] = h;
        H[(size_t)cell * n * n + b * n + a] = h;
    }
}

__global__ void isotropic_kernel(int n, double m0, const double *__restrict__ u,
                                 double *__restrict__ alpha, int C)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        const double u0 = u[(size_t)c * n];
        alpha[(size_t)c * n] = log(u0 / (4.0 * 3.14159265358979323846 * m0)) / m0;
        for (int a = 1; a < n; ++a) alpha[(size_t)c * n + a] = 0.0;
    }
}

__global__ void ansatz_kernel(Tables T, const double *__restrict__ alpha, double *__restrict__ psi,
                              int C)
{
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int n = T.n, Qp = T.Qp, Qf = T.Qf;
    for (int cell = blockIdx.x * kWarps + wib; cell < C; cell += gridDim.x * kWarps) {
        for (int q = lane; q < Qf; q += 32) {
            double z = 0.0;
            for (int b = 0; b < n; ++b) z = fma(alpha[(size_t)cell * n + b], T.Mt[b * Qp + q], z);
            psi[(size_t)cell * Qf + q] = kexp(z, T.exptab);
        }
    }
}

int grid_for(const kitrt_mn *mn, int C, int per_sm)
{
    const int need = (C + kWarps - 1) / kWarps;
    const int cap = mn->nsm * per_sm;
    return need < cap ? (need > 0 ? need : 1) : cap;
}

template <int NN, bool SEG = false>
int predict_launch(kitrt_mn *mn, const NewtonState &S, int C, const double *u, NewtonParams np,
                   const int32_t *list, const int32_t *count, cudaStream_t s)
{
    using D = PredictDims<NN, SEG>;
    // the factors of more cells than three warps on every SM hold: in segments
    if constexpr (NN == 5 && !SEG)
        if (C > mn->nsm * 3 * 32) return predict_launch<NN, true>(mn, S, C, u, np, list, count, s);
    if (ensure_dyn_smem(predict_kernel<NN, SEG>, D::smem)) return KITRT_ECUDA;
    int tb = (C + D::threads - 1) / D::threads;
    if (tb > mn->nsm * 32) tb = mn->nsm * 32;
    predict_kernel<NN, SEG><<<tb > 0 ? tb : 1, D::threads, D::smem, s>>>(S, u, np, list, count);
    return KITRT_OK;
}

}  // namespace

#define KITRT_DISPATCH_N(N, ...)                        \
    switch (N) {                                        \
    case 1: { constexpr int NN = 1; __VA_ARGS__; } break; \
    case 2: { constexpr int NN = 2; __VA_ARGS__; } break; \
    case 3: { constexpr int NN = 3; __VA_ARGS__; } break; \
    case 4: { constexpr int NN = 4; __VA_ARGS__; } break; \
    case 5: { constexpr int NN = 5; __VA_ARGS__; } break; \
    default: return KITRT_EINVAL;                       \
    }

int launch_isotropic(const Tables &T, int C, const double *u, double *alpha, cudaStream_t s)
{
    const int blocks = (C + 255) / 256;
    isotropic_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(T.n, T.m0, u, alpha, C);
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// Cells up to which a round of the FP64 mode goes to the 8-lane kernel (N <= 3): there a warp's FP64
// instructions serve 4 cells instead of 32, which is slower once the thread-per-cell kernel has warps for
// the SMs. M_3, whole passes with the line at 8,192 and at 14,000 cells: 20,001 closures of 24 rounds
// 2.385 and 2.416 ms, adjoint of 59,168 cells 41.65 and 41.78 ms.
constexpr int kGroupUpTo = 8192;

// Newton step of the listed cells.
int launch_post(kitrt_mn *mn, const Tables &T, const NewtonState &S, int C, const double *u, int k,
                NewtonParams np, double *Vacc, cudaStream_t s)
{
    const bool mixed = mn->p.mode != KITRT_FP64;
    const int upto = mixed || mn->N > 3 ? 0x7fffffff : kGroupUpTo;
    const int nu64 = units64(mn->R * mn->J), nunits = mixed ? mn->Qs / 32 : nu64;
    const int sweep_grid = mixed ? mn->grid_mixed : mn->grid_fp64, target = mixed ? mn->target_mixed : mn->target_fp64;
    if (C > upto) {
        // 64-thread blocks: small blocks spread the listed cells over every SM
        int blocks = (C + kPostBlock - 1) / kPostBlock;
        if (blocks > mn->nsm * 32) blocks = mn->nsm * 32;
        const size_t smem = post_smem_bytes(mn->n, mn->n2, mn->npairs, mn->gaunt_nnz);
        LaunchScope ls(mn, PK_POST, s, 0);
        int rc = KITRT_OK;
#define THREAD_CASE(NNv)                                                                                       \
    case NNv:                                                                                                  \
        rc = ensure_dyn_smem(post_thread_kernel<NNv>, smem);                                                   \
        if (!rc)                                                                                               \
            post_thread_kernel<NNv><<<blocks, kPostBlock, smem, s>>>(T, S, u, k, np, Vacc, mn->vs,             \
                                                                     mn->gaunt_nnz, sweep_grid, target,        \
                                                                     nunits, upto);                            \
        break;
        switch (mn->N) {
            THREAD_CASE(1)
            THREAD_CASE(2)
            THREAD_CASE(3)
        default: return KITRT_EINVAL;
        }
#undef THREAD_CASE
        if (rc) return rc;
        if (cudaGetLastError() != cudaSuccess) return KITRT_ECUDA;
    }
    const size_t smem = group_smem_bytes(mn->n2, mn->npairs, mn->gaunt_nnz, mixed);
    int blocks = (C + kGroupCells - 1) / kGroupCells;
    const int most = mn->nsm * (mn->N > 3 ? 2 : 4);
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    LaunchScope ls(mn, PK_POST, s, 0);
    int rc = KITRT_OK;
    if (mixed) {
        KITRT_DISPATCH_N(mn->N, rc = ensure_dyn_smem(post_group_kernel<NN, true>, smem));
        if (rc) return rc;
        KITRT_DISPATCH_N(mn->N, (post_group_kernel<NN, true><<<blocks, kGroupBlock, smem, s>>>(T, S, u, k, np, Vacc, mn->vs, mn->vs_handed, mn->gaunt_nnz, sweep_grid, target, nunits, mn->grid_fp64, mn->target_fp64, nu64, upto)));
    } else {
        KITRT_DISPATCH_N(mn->N, rc = ensure_dyn_smem(post_group_kernel<NN, false>, smem));
        if (rc) return rc;
        KITRT_DISPATCH_N(mn->N, (post_group_kernel<NN, false><<<blocks, kGroupBlock, smem, s>>>(T, S, u, k, np, Vacc, mn->vs, mn->vs_handed, mn->gaunt_nnz, sweep_grid, target, nunits, mn->grid_fp64, mn->target_fp64, nu64, upto)));
    }
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int launch_moments_fp64(kitrt_mn *mn, const Tables &T, int C, const double *alpha, double *V, cudaStream_t s)
{
    const int grid = grid_for(mn, C, 8);
    LaunchScope ls(mn, PK_OTHER, s, C);
    KITRT_DISPATCH_N(mn->N, moments_kernel<NN><<<grid, kWarps * 32, 0, s>>>(T, alpha, V, C));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int launch_gaunt(kitrt_mn *mn, const Tables &T, int C, const double *V, double *H, cudaStream_t s)
{
    const long total = (long)C * (T.n * (T.n + 1) / 2);
    int blocks = (int)((total + 255) / 256);
    if (blocks > mn->nsm * 16) blocks = mn->nsm * 16;
    LaunchScope ls(mn, PK_OTHER, s, C);
    gaunt_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(T, V, H, C);
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int launch_ansatz(const Tables &T, int C, const double *alpha, double *psi, cudaStream_t s)
{
    const int blocks = (C + kWarps - 1) / kWarps;
    ansatz_kernel<<<blocks > 0 ? blocks : 1, kWarps * 32, 0, s>>>(T, alpha, psi, C);
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int launch_begin(kitrt_mn *mn, const Tables &T, const NewtonState &S, int C,
                 const double *u, const double *alpha_in, int first, NewtonParams np,
                 cudaStream_t s, int learned, int renew)
{
    (void)T;
    int blocks = (C + 255) / 256;
    if (blocks > mn->nsm * 8) blocks = mn->nsm * 8;
    {
        LaunchScope ls(mn, PK_BEGIN, s, C);
        KITRT_DISPATCH_N(mn->N, begin_test_kernel<NN><<<blocks > 0 ? blocks : 1, 256, 0, s>>>(S, u, alpha_in, first, np, C, learned, renew));
        if (cudaGetLastError() != cudaSuccess) return KITRT_ECUDA;
    }
    if (first == 1 || learned) return KITRT_OK;
    return launch_predict(mn, S, C, u, np, S.list[1], S.cnt + 8, s);
}

// The first Newton step of the cells in `list` (device, *count of them, at most C) from their stored
// moments and factors.
int launch_predict(kitrt_mn *mn, const NewtonState &S, int C, const double *u, NewtonParams np, const int32_t *list,
                   const int32_t *count, cudaStream_t s)
{
    LaunchScope ls(mn, PK_BEGIN, s, 0);
    int rc = KITRT_OK;
    KITRT_DISPATCH_N(mn->N, rc = predict_launch<NN>(mn, S, C, u, np, list, count, s));
    if (rc) return rc;
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// Grid of the FP64 sweep: as many CTAs as are resident on all SMs at once.
int fp64_sweep_grid(const kitrt_mn *mn)
{
    const size_t smem = sweep64_smem(mn->n, mn->n2, mn->N, mn->J);
    int resident = 1;
#define GRID_CASE(NNv)                                                              \
    case NNv:                                                                       \
        if (ensure_dyn_smem(sweep64_kernel<NNv, Cells::kListed>, smem)) return mn->nsm;             \
        resident = resident_ctas(sweep64_kernel<NNv, Cells::kListed>, kSweepThreads, smem, 8);      \
        break;
    switch (mn->N) {
        GRID_CASE(1)
        GRID_CASE(2)
        GRID_CASE(3)
        GRID_CASE(4)
        GRID_CASE(5)
    default: break;
    }
#undef GRID_CASE
    return mn->nsm * resident;
}

int launch_eval_fp64(kitrt_mn *mn, const Tables &T, const NewtonState &S, const double *u, int k, cudaStream_t s)
{
    LaunchScope ls(mn, PK_EVAL, s, 0);
    const size_t smem = sweep64_smem(mn->n, mn->n2, mn->N, mn->J);
    int rc = KITRT_OK;
    KITRT_DISPATCH_N(mn->N, rc = ensure_dyn_smem(sweep64_kernel<NN, Cells::kListed>, smem));
    if (rc) return rc;
    KITRT_DISPATCH_N(mn->N, (sweep64_kernel<NN, Cells::kListed><<<mn->grid_fp64, kSweepThreads, smem, s>>>(T, S, u, k, mn->d_Vacc, mn->vs, mn->target_fp64, nullptr, nullptr, 0)));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// Mixed modes: the cells handed over to the FP64 Hessian in earlier rounds. They are few (often none)
// and lie side by side in the list, so they are swept from a list of their own, split over as many
// parts as fill the SMs (a warp per flagged entry of the list took 0.3 to
// 0.8 ms a round for a handful of M_5 cells, and 1.19 of 2.8 ms of a checkerboard step).
int launch_eval_handed(kitrt_mn *mn, const Tables &T, const NewtonState &S, const double *u, int k, float *psi32,
                       cudaStream_t s)
{
    LaunchScope ls(mn, PK_EVAL, s, 0);
    const size_t smem = sweep64_smem(mn->n, mn->n2, mn->N, mn->J);
    int rc = KITRT_OK;
    KITRT_DISPATCH_N(mn->N, rc = ensure_dyn_smem(sweep64_kernel<NN, Cells::kHanded>, smem));
    if (rc) return rc;
    KITRT_DISPATCH_N(mn->N, (sweep64_kernel<NN, Cells::kHanded><<<mn->grid_fp64, kSweepThreads, smem, s>>>(T, S, u, k, mn->d_Vacc, mn->vs, mn->target_fp64, nullptr, psi32, mn->vs_handed)));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// The allocation-free closure's round (the caller passes a launch-only view without a mesh).
int launch_eval_fused(kitrt_mn *mn, const Tables &T, const NewtonState &S, int C, const double *u, int k,
                      NewtonParams np, cudaStream_t s)
{
    const int grid = grid_for(mn, C, 4);
    LaunchScope ls(mn, PK_EVAL, s, 0);
    KITRT_DISPATCH_N(mn->N, (eval_kernel<NN><<<grid, kWarps * 32, 0, s>>>(T, S, u, k, np)));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

// Degree-2N moments (columns of V, stride vs) and FP64 ansatz of every cell at the given alphas, whose
// zeroth moments are about u's.
int launch_adjoint_closure(kitrt_mn *mn, const Tables &T, int C, const double *u, const double *alpha, double *V,
                           int vs, double *psi, cudaStream_t s)
{
    const size_t smem = sweep64_smem(mn->n, mn->n2, mn->N, mn->J);
    const int tiles = (C + kSweepThreads - 1) / kSweepThreads;
    const NewtonState S{};
    int rc = KITRT_OK;
    KITRT_DISPATCH_N(mn->N, rc = ensure_dyn_smem(sweep64_kernel<NN, Cells::kGiven>, smem));
    if (rc) return rc;
    LaunchScope ls(mn, PK_ADJOINT, s, C);
    KITRT_DISPATCH_N(mn->N, (sweep64_kernel<NN, Cells::kGiven><<<std::min(tiles, mn->grid_fp64), kSweepThreads, smem, s>>>(T, S, u, 0, V, vs, 0, alpha, psi, C)));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}

int launch_finish(kitrt_mn *mn, const Tables &T, const NewtonState &S, int C,
                  double *alpha_out, double *psi, int polish, int compare_prev, cudaStream_t s)
{
    LaunchScope ls(mn, PK_FINISH, s, C);
    if (!psi) {
        const size_t total = (size_t)C * T.n;
        int blocks = (int)((total + 255) / 256);
        if (blocks > mn->nsm * 8) blocks = mn->nsm * 8;
        finish_alpha_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(S, alpha_out, polish, T.n, C);
        return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
    }
    const size_t smem = 2048 * 8 + (size_t)T.J * 2 * mn->N * 8 + (size_t)T.n * 32 * 8 + kFinishWarps * 32 * 8;
    int blocks = (C + 31) / 32;
    if (blocks > mn->nsm * 16) blocks = mn->nsm * 16;
    KITRT_DISPATCH_N(mn->N, finish_kernel<NN><<<blocks > 0 ? blocks : 1, kFinishWarps * 32, smem, s>>>(T, S, alpha_out, psi, polish, compare_prev, C));
    return cudaGetLastError() == cudaSuccess ? KITRT_OK : KITRT_ECUDA;
}
