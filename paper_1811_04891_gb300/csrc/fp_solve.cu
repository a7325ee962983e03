// fp_solve.cu -- everything of the location stage that is compiled per order
// (Sec. 2.1): the Newton kernels, the classification and their launch
// sequence, for n = FP_N GLL points per direction.  One object per order, so
// that the orders build in parallel.
//
// Where is_tile_order says so, the tensor-core tile kernels (fp_tile.cuh) run
// in every entry point and at every number of pairs: a pair's result does not
// depend on the pairs it shares a warp with, so all entry points agree bit
// for bit.  The other orders keep one thread per pair.
#include <algorithm>
#include <atomic>

#include "fp_common.cuh"
#include "fp_internal.h"
#include "fp_newton.cuh"
#include "fp_rank.cuh"
#include "fp_tile_launch.cuh"

#ifndef FP_N
#error "FP_N: GLL points per direction"
#endif

namespace fpg {

#define FP_CAT2(a, b) a##b
#define FP_CAT(a, b) FP_CAT2(a, b)

// the mixed form's tile kernels (fp_tile_mixed.cu)
cudaError_t FP_CAT(newton_tile_mixed_, FP_N)(const FindArgs& a, const NewtonArgs& na, int64_t npairs, const BasisTab& tab,
                                             int block, unsigned grid, cudaStream_t s);
int FP_CAT(tile_fit_mixed_, FP_N)(int block);
cudaError_t FP_CAT(digits_mixed_, FP_N)(int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig,
                                        const BasisTab& tab, cudaStream_t s);

// ---------------------------------------------------------------------------
// Newton kernels, one thread per pair (the solver is in fp_newton.cuh)
// ---------------------------------------------------------------------------
// FP64 form: nearest-node (or warm) start, full FP64 trust-region Newton;
// with A.pstate, the first pass stops a solve after A.first_pass iterations
// and lists it (fbl, capacity fbc) for the second.  Measured on the 32^3
// N=7 workload: budgets 1 / 2 / 3 / 4 / 5 / 6 gave 387 / 300 / 311 / 319 /
// 323 / 326 ms for the two passes together; the batch's per-order groups
// measured faster with 4 (82 / 88 ms for N = 5 / 7 against 105 / 104 with 2).
constexpr int kFirstPass = 2;
constexpr int kFirstPassBatch = 4;

template <int n>
__device__ __forceinline__ void solve_pair(const NewtonArgs& A, const BasisTab& tab, int64_t s, int32_t* fbl,
                                           int64_t fbc)
{
    constexpr int n3 = n * n * n;
    const int32_t q = A.order[s];
    const int e = A.pair_elem[q] - A.ebase;
    const int64_t p = pair_point(A.pair_pt[q]);
    const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
    const ElemPtr<double> el64 = {A.coords + (int64_t)e * n3, A.coords + (A.E + e) * n3,
                                  A.coords + (2 * A.E + e) * n3};
    double r[3], J[9];
    if (!warm_seed(A, p, e, r)) seed_nearest<n, double>(el64, tab, xs, r);
    bool conv64;
    NewtonState st{1.0, 0, 0, false};
    const double res = newton<n, double, true>(el64, tab, xs, r, J, A.max_newton, conv64, A.pstate ? &st : nullptr,
                                               A.first_pass);
    const int64_t w = result_slot(A, s, q);
    A.prst[w] = r[0];
    A.prst[A.cap + w] = r[1];
    A.prst[2 * A.cap + w] = r[2];
    if (st.paused) {
        // still iterating after the first pass's budget: continued by
        // k_newton_resume, so that warps of the first pass do not wait on it
        A.pres[w] = -1.0;
        A.pstate[w] = make_double2(st.rho, (double)(st.chord_fail + 4 * st.it));
        const int32_t k = atomicAdd(A.fb_count, 1);
        if (k < fbc) fbl[k] = (int32_t)w;
    } else {
        A.pres[w] = res;
    }
}

// pass 2 of the FP64 form: the solves paused by the first pass, resumed
// where they stopped, one per thread (the list is dense: every lane has a
// long solve).  If the list overflowed, the paused slots (pres < 0) are
// found by scanning the range instead.
template <int n>
__device__ __forceinline__ void resume_pair(const NewtonArgs& A, const BasisTab& tab, int64_t w)
{
    constexpr int n3 = n * n * n;
    const int32_t q = listed_pair(A, w);
    const int e = A.pair_elem[q] - A.ebase;
    const int64_t p = pair_point(A.pair_pt[q]);
    const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
    const ElemPtr<double> el64 = {A.coords + (int64_t)e * n3, A.coords + (A.E + e) * n3,
                                  A.coords + (2 * A.E + e) * n3};
    double r[3] = {A.prst[w], A.prst[A.cap + w], A.prst[2 * A.cap + w]}, J[9];
    const double2 sv = A.pstate[w];
    const int code = (int)sv.y;
    NewtonState st{sv.x, code & 3, code >> 2, false};
    bool conv;
    const double res = newton<n, double, true>(el64, tab, xs, r, J, A.max_newton, conv, &st);
    A.prst[w] = r[0];
    A.prst[A.cap + w] = r[1];
    A.prst[2 * A.cap + w] = r[2];
    A.pres[w] = res;
}

template <int n>
__global__ void __launch_bounds__(128) k_newton_resume(NewtonArgs A, BasisTab tab)
{
    const PairRange R = pair_range(A);
    const int32_t* fbl = A.fb_list + (A.s_lo ? R.s0 : 0);
    const int64_t fbc = A.s_lo ? R.s1 - R.s0 : A.fb_cap;
    const int64_t nfb = *A.fb_count;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, dt = (int64_t)gridDim.x * blockDim.x;
    if (nfb <= fbc) {
        for (int64_t t = t0; t < nfb; t += dt) resume_pair<n>(A, tab, fbl[t]);
    } else {
        for (int64_t s = R.s0 + t0; s < R.s1; s += dt) {
            const int64_t w = result_slot(A, s, A.order[s]);
            if (A.pres[w] < 0.0) resume_pair<n>(A, tab, w);
        }
    }
}

// passes 1 and 2 in one kernel: the FP32 work of some warps overlaps the
// FP64 work of others (the orders without a tile kernel).
// Its launch shape.  CAP (blocks of up to 128 threads, n <= 10, where 128
// registers need no spills): registers capped so that four blocks of 128
// threads fit an SM.  Otherwise (persistent grids of the workspace calls,
// larger n) the compiler takes what it wants, 222 registers at n = 13; that
// has to be asked for by the block count: left out, 128 are used and a find
// of 10,000 points in 512 elements of order 12 takes 960 us instead of 838.
template <int n, bool CAP> struct MixedLB {
    static constexpr int threads = CAP ? 128 : 256;
    static constexpr int blocks = CAP ? 4 : 1;
};

template <int n>
__device__ __forceinline__ void solve_mixed(const NewtonArgs& A, const BasisTab& tab, int64_t s, int32_t* fbl,
                                            int64_t fbc)
{
    constexpr int n3 = n * n * n;
    {
        const int32_t q = A.order[s];
        const int e = A.pair_elem[q] - A.ebase;
        const int64_t p = pair_point(A.pair_pt[q]);
        const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
        const double* c = A.boxes[e].c;
        const double xd[3] = {xs[0] - c[0], xs[1] - c[1], xs[2] - c[2]};
        const float xl[3] = {(float)xd[0], (float)xd[1], (float)xd[2]};
        const ElemPtr<float> el32 = {A.coords32 + (int64_t)e * n3, A.coords32 + (A.E + e) * n3,
                                     A.coords32 + (2 * A.E + e) * n3};
        float r32[3], J32[9];
        {
            double rw[3];
            if (warm_seed(A, p, e, rw)) {
                r32[0] = (float)rw[0]; r32[1] = (float)rw[1]; r32[2] = (float)rw[2];
            } else {
                seed_nearest<n, float>(el32, tab, xl, r32);
            }
        }
        bool conv32;
        const float res32 = newton<n, float, false>(el32, tab, xl, r32, J32, A.max_newton, conv32);
        double r[3] = {r32[0], r32[1], r32[2]};
        double res = conv32 ? (double)res32 : -1.0;
        if (A.stats) {
            if (!conv32) atomicAdd(A.stats + 1, 1ULL);
            else if ((double)res32 > A.reject32 * A.boxes[e].he) atomicAdd(A.stats + 0, 1ULL);
        }
        if (conv32 && (double)res32 <= A.reject32 * A.boxes[e].he) {
            // Final Newton steps at FP64 accuracy: compensated (double-float)
            // residuals on the split element-local coordinates, on the FP32
            // pipes, with the FP32 Jacobian and the active-set step.  A step
            // that is still large is taken as computed in FP32; once it is
            // small, the 3x3 solve is repeated in FP64, and an FP64 step within
            // the tolerance confirms convergence: r is kept with its own
            // residual (as in chord64).  An FP64 step s above the tolerance ct
            // but at most kTake * ct is taken, and the residual at r + s is
            // the linear model f + J s: the Jacobian (FP32, from the last FP32
            // iterate) has a relative error eps of at most ~1e-4, so r + s is
            // within eps |s| <= 0.1 ct of the solution and f + J s within
            // eps |J s| of its residual -- a further compensated residual
            // would only confirm this.  Unconfirmed after A.refine residuals:
            // the pair goes to the full FP64 Newton.
            const ElemPtr<float> lo32 = {A.coords32lo + (int64_t)e * n3, A.coords32lo + (A.E + e) * n3,
                                         A.coords32lo + (2 * A.E + e) * n3};
            res = -1.0;
            for (int it = 0; it < A.refine; ++it) {
                float f[3], d32[3];
                resid_df<n>(el32, lo32, tab, r, xd, f);
                const double fd[3] = {(double)f[0], (double)f[1], (double)f[2]};
                if (f[0] == 0.0f && f[1] == 0.0f && f[2] == 0.0f) {   // exact hit
                    res = 0.0;
                    break;
                }
                // the active set is decided on r itself: a coordinate just inside
                // a bound must not round onto it (it would be frozen off the bound)
                const float rf[3] = {f32_inside(r[0]), f32_inside(r[1]), f32_inside(r[2])};
                if (gn_step<float>(J32, f, rf, d32) == 0) {  // KKT point at a vertex
                    res = sqrt(fd[0] * fd[0] + fd[1] * fd[1] + fd[2] * fd[2]);
                    break;
                }
                double d[3] = {(double)d32[0], (double)d32[1], (double)d32[2]};
                const bool small = fmaxf(fabsf(d32[0]), fmaxf(fabsf(d32[1]), fabsf(d32[2]))) <= (float)kConfirm;
                if (small) {
                    double J[9];
#pragma unroll
                    for (int k = 0; k < 9; ++k) J[k] = (double)J32[k];
                    if (gn_step<double>(J, fd, r, d) == 0) {
                        res = sqrt(fd[0] * fd[0] + fd[1] * fd[1] + fd[2] * fd[2]);
                        break;
                    }
                    double rn[3];
                    box_step<double>(r, d, rn);
                    const double sn = fmax(fabs(rn[0] - r[0]), fmax(fabs(rn[1] - r[1]), fabs(rn[2] - r[2])));
                    const double ct = chord_tol_df(J, A.boxes[e].he);
                    if (sn <= ct) {
                        res = sqrt(fd[0] * fd[0] + fd[1] * fd[1] + fd[2] * fd[2]);
                        break;
                    }
                    if (sn <= kTake * ct) {
                        double g[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            g[a] = fd[a] + J[3 * a] * (rn[0] - r[0]) + J[3 * a + 1] * (rn[1] - r[1]) +
                                   J[3 * a + 2] * (rn[2] - r[2]);
                        r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                        res = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
                        break;
                    }
                    r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                } else {
                    double rn[3];
                    box_step<double>(r, d, rn);
                    r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                }
            }
            if (A.stats) atomicAdd(A.stats + (res < 0.0 ? 3 : 2), 1ULL);
        }
        const int64_t w = result_slot(A, s, q);
        A.prst[w] = r[0];
        A.prst[A.cap + w] = r[1];
        A.prst[2 * A.cap + w] = r[2];
        A.pres[w] = res;
        if (res < 0.0) {
            const int32_t k = atomicAdd(A.fb_count, 1);
            if (k < fbc) fbl[k] = (int32_t)w;
        }
    }
}

template <int n, bool CAP>
__global__ void __launch_bounds__(MixedLB<n, CAP>::threads, MixedLB<n, CAP>::blocks)
    k_newton_mixed(NewtonArgs A, BasisTab tab)
{
    const PairRange R = pair_range(A);
    int32_t* fbl = A.fb_list + (A.s_lo ? R.s0 : 0);
    const int64_t fbc = A.s_lo ? R.s1 - R.s0 : A.fb_cap;
    for_each_pair(A, R, [&](int64_t s) { solve_mixed<n>(A, tab, s, fbl, fbc); });
}

// pass 3 (FP64): full trust-region Newton for the pairs marked -1, from the
// point the earlier passes reached.  These pairs are few and scattered, and
// each solve is a long dependent chain: the kernel is latency-bound.  The
// mixed pass listed them (fb_list); each block is one warp and solves one
// listed pair at a time with the warp-cooperative evaluators, which shortens
// the chain about 16-fold.  If the list overflowed, blocks instead gather the
// marked pairs of chunks of slots into shared memory and solve those one per
// lane.
constexpr int kFullChunk = 8192;
constexpr int kFullSub = 1024;

template <int n>
__device__ __forceinline__ void solve_full64(const NewtonArgs& A, const BasisTab& tab, int64_t w)
{
    constexpr int n3 = n * n * n;
    const int32_t q = listed_pair(A, w);
    const int e = A.pair_elem[q] - A.ebase;
    const int64_t p = pair_point(A.pair_pt[q]);
    const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
    const ElemPtr<double> el64 = {A.coords + (int64_t)e * n3, A.coords + (A.E + e) * n3,
                                  A.coords + (2 * A.E + e) * n3};
    double r[3] = {A.prst[w], A.prst[A.cap + w], A.prst[2 * A.cap + w]}, J[9];
    bool conv;
    const double res = newton<n, double, true>(el64, tab, xs, r, J, A.max_newton, conv);
    A.prst[w] = r[0];
    A.prst[A.cap + w] = r[1];
    A.prst[2 * A.cap + w] = r[2];
    A.pres[w] = res;
}

template <int n>
__global__ void __launch_bounds__(32) k_newton64_full(NewtonArgs A, BasisTab tab)
{
    const PairRange R = pair_range(A);
    const int32_t* fbl = A.fb_list + (A.s_lo ? R.s0 : 0);
    const int64_t fbc = A.s_lo ? R.s1 - R.s0 : A.fb_cap;
    const int64_t nfb = *A.fb_count;
    if (nfb <= fbc) {
        // one warp (this block) per listed pair
        constexpr int n3 = n * n * n;
        for (int64_t t = blockIdx.x; t < nfb; t += gridDim.x) {
            const int64_t w = fbl[t];
            const int32_t q = listed_pair(A, w);
            const int e = A.pair_elem[q] - A.ebase;
            const int64_t p = pair_point(A.pair_pt[q]);
            const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
            const ElemPtr<double> el64 = {A.coords + (int64_t)e * n3, A.coords + (A.E + e) * n3,
                                          A.coords + (2 * A.E + e) * n3};
            double r[3] = {A.prst[w], A.prst[A.cap + w], A.prst[2 * A.cap + w]}, J[9];
            bool conv;
            const double res = newton<n, double, true, true>(el64, tab, xs, r, J, A.max_newton, conv);
            if (threadIdx.x == 0) {
                A.prst[w] = r[0];
                A.prst[A.cap + w] = r[1];
                A.prst[2 * A.cap + w] = r[2];
                A.pres[w] = res;
            }
        }
        return;
    }
    __shared__ int32_t list[kFullSub];
    __shared__ int count;
    for (int64_t base = R.s0 + (int64_t)blockIdx.x * kFullChunk; base < R.s1; base += (int64_t)gridDim.x * kFullChunk) {
        const int64_t cend = base + kFullChunk < R.s1 ? base + kFullChunk : R.s1;
        for (int64_t sb = base; sb < cend; sb += kFullSub) {
            if (threadIdx.x == 0) count = 0;
            __syncthreads();
            const int64_t end = sb + kFullSub < cend ? sb + kFullSub : cend;
            for (int64_t s = sb + threadIdx.x; s < end; s += blockDim.x) {
                const int64_t w = result_slot(A, s, A.order[s]);
                if (A.pres[w] < 0.0) list[atomicAdd(&count, 1)] = (int32_t)w;
            }
            __syncthreads();
            const int m = count;
            for (int t = threadIdx.x; t < m; t += blockDim.x) solve_full64<n>(A, tab, list[t]);
            __syncthreads();
        }
    }
}

template <int n>
__global__ void __launch_bounds__(256) k_newton(NewtonArgs A, BasisTab tab)
{
    const PairRange R = pair_range(A);
    int32_t* fbl = A.fb_list + (A.s_lo ? R.s0 : 0);
    const int64_t fbc = A.s_lo ? R.s1 - R.s0 : A.fb_cap;
    for_each_pair(A, R, [&](int64_t s) { solve_pair<n>(A, tab, s, fbl, fbc); });
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// grid for `work` items; with a persistent block count the kernels loop
// grid-stride over a count that only the device knows
static unsigned grid_for(int64_t work, int block, int persistent)
{
    int64_t g = (work + block - 1) / block;
    if (persistent > 0 && g > persistent) g = persistent;
    return (unsigned)(g < 1 ? 1 : g);
}

// Newton stage (and the mixed form's FP64 fallback) over the pairs of a:
// all live pairs, or (batch groups, a.s_lo set) the group's sorted range.
// grid == 0: sized from npairs and the block (persistent when the caller
// gave persistent_blocks).
template <int n, bool MIXED>
static cudaError_t newton_form(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp, int block,
                               unsigned grid, cudaStream_t s)
{
    NewtonArgs na;
    na.dcount = a.off + a.P;
    na.E = a.E;
    na.order = a.order;
    na.pair_elem = a.pair_elem;
    na.pair_pt = a.pair_pt;
    na.P = a.P;
    na.pts = a.pts;
    na.coords = a.coords;
    na.coords32 = a.coords32;
    na.coords32lo = a.coords32lo;
    na.boxes = a.boxes;
    na.pres = a.pres;
    na.prst = a.prst;
    na.cap = a.cap;
    na.reject32 = 1e-4;
    na.max_newton = fp.max_newton;
    na.refine = fp.refine;
    na.first_pass = a.batch ? kFirstPassBatch : kFirstPass;
    na.stats = a.stats;
    na.warm_elem = a.warm_elem;
    na.warm_rst = a.warm_rst;
    na.fb_count = nullptr;
    na.fb_list = nullptr;
    na.fb_cap = 0;
    na.s_lo = a.s_lo;
    na.s_hi = a.s_hi;
    na.ebase = a.ebase;
    na.queue = a.queue;
    na.tile = a.tile > 0 ? a.tile : block;
    na.pstate = nullptr;
    na.walk = a.inv != nullptr;
    na.digits = a.digits;
    na.pause_list = nullptr;
    na.pause_count = nullptr;
    na.resume = false;
    na.list_blocks = 0;
    na.list_spread = 0;
    na.jst = nullptr;
    na.rows = 32;
    cudaError_t err;
    if (a.queue && (err = cudaMemsetAsync(a.queue, 0, sizeof(int32_t), s)) != cudaSuccess) return err;
    if (MIXED || !is_tile_order(n, MIXED)) {
        if (a.s_lo) {
            // batch group: its own counter; its list from the group's first sorted position
            na.fb_count = a.fb_count;
            na.fb_list = a.fb_list;
        } else {
            // list of left-over pairs: the per-point counts (free after the scan) hold
            // the slots, the first scan scratch word (free after the sort) the count
            na.fb_count = a.scan_tmp;
            na.fb_list = a.cnt;
            na.fb_cap = a.P;
        }
        if (MIXED || a.pstate)
            if ((err = cudaMemsetAsync(na.fb_count, 0, sizeof(int32_t), s)) != cudaSuccess) return err;
    }
    if constexpr (is_tile_order(n, MIXED)) {
        if constexpr (MIXED) err = FP_CAT(newton_tile_mixed_, FP_N)(a, na, npairs, tab, block, grid, s);
        else err = newton_tile<n, false>(a, na, npairs, tab, block, grid, s);
        if (err != cudaSuccess) return err;
    } else {
        if (grid == 0) grid = grid_for(npairs, block, a.persistent_blocks);
        if constexpr (MIXED) {
            bool capped = false;
            if constexpr (n <= 10) {
                if (block <= 128 && (a.persistent_blocks == 0 || a.queue)) {
                    k_newton_mixed<n, true><<<grid, block, 0, s>>>(na, tab);
                    capped = true;
                }
            }
            if (!capped) k_newton_mixed<n, false><<<grid, block, 0, s>>>(na, tab);
        } else {
            na.pstate = a.pstate;
            k_newton<n><<<grid, block, 0, s>>>(na, tab);
            // the resumed solves: one per thread over the list (at most the
            // pairs of the first pass), sized like the first pass's grid
            if (a.pstate) {
                k_newton_resume<n><<<std::max(1u, grid / 2), 128, 0, s>>>(na, tab);
                count_launch();
            }
        }
        count_launch();
    }
    if constexpr (MIXED) {
        // blocks of one warp: enough for a list of up to 38,912 pairs in one
        // pass, and for the chunked path over every slot if it overflowed
        const unsigned gfull = (unsigned)std::max<int64_t>(
            1216, a.persistent_blocks > 0 || a.s_lo ? 0 : (npairs + kFullChunk - 1) / kFullChunk);
        k_newton64_full<n><<<gfull, 32, 0, s>>>(na, tab);
        count_launch();
    }
    return cudaGetLastError();
}

template <int n>
static cudaError_t newton_n(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp, int block,
                            unsigned grid, cudaStream_t s)
{
    return fp.mixed ? newton_form<n, true>(a, npairs, tab, fp, block, grid, s)
                    : newton_form<n, false>(a, npairs, tab, fp, block, grid, s);
}

template <int n>
static cudaError_t solve_n(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp, int block,
                           cudaStream_t s)
{
    if (npairs > 0) {
        if (a.ev[2]) cudaEventRecord(a.ev[2], s);
        if (a.persistent_blocks == 0 && !is_tile_order(n, fp.mixed)) block = spread_block(npairs, block);
        cudaError_t err = newton_n<n>(a, npairs, tab, fp, block, 0, s);
        if (err != cudaSuccess) return err;
        if (a.ev[3]) cudaEventRecord(a.ev[3], s);
    }
    RankArgs ra;
    ra.P = a.P;
    ra.E = a.E;
    ra.off = a.off;
    ra.pair_elem = a.pair_elem;
    ra.pres = a.pres;
    ra.prst = a.prst;
    ra.cap = a.cap;
    ra.sub = a.sub;
    ra.boxes = a.boxes;
    ra.dist = a.dist;
    ra.code = a.code;
    ra.osub = a.osub;
    ra.oelem = a.oelem;
    ra.rst = a.rst;
    ra.dist2 = a.dist2;
    ra.pair_pt = a.pair_pt;
    ra.F = a.eval.F;
    ra.out = a.eval.out;
    ra.band = a.band;
    ra.inv = a.inv;
    if (a.ev[4]) cudaEventRecord(a.ev[4], s);
    k_rank<n, 3><<<(unsigned)((a.P + kRankThreads - 1) / kRankThreads), kRankThreads, 0, s>>>(ra, fp, tab);
    count_launch();
    if (a.ev[5]) cudaEventRecord(a.ev[5], s);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || a.eval.F == 0 || npairs == 0) return err;
    if (a.ev[6]) cudaEventRecord(a.ev[6], s);
    err = launch_eval_pairs(n, a.E, a.P, a.off + a.P, a.cap, a.order, a.pair_elem, a.pair_pt, a.prst, a.eval, tab,
                            grid_for(npairs, 128, a.persistent_blocks ? 4 * a.persistent_blocks : 0), s, nullptr,
                            nullptr, 0, a.inv != nullptr);
    if (a.ev[7]) cudaEventRecord(a.ev[7], s);
    return err;
}

// Blocks of `block` threads of the Newton kernel a group of order n - 1
// would launch (find_newton_group) that fit one SM at once.
template <int n, bool MIXED>
static int newton_fit_form(int block)
{
    if constexpr (is_tile_order(n, MIXED)) {
        if constexpr (MIXED) return FP_CAT(tile_fit_mixed_, FP_N)(std::min(block, 128));
        else return tile_fit<n, TILE_FP64>(std::min(block, 128));
    } else {
        int k = 0;
        cudaError_t e;
        if constexpr (MIXED)
            e = block <= 128 && n <= 10 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_newton_mixed<n, n <= 10>, block, 0)
                                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_newton_mixed<n, false>, block, 0);
        else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_newton<n>, block, 0);
        return e == cudaSuccess ? k : 1;
    }
}

template <int n>
static int newton_fit(bool mixed, int block)
{
    return mixed ? newton_fit_form<n, true>(block) : newton_fit_form<n, false>(block);
}

template <int n, bool MIXED>
static cudaError_t digits_if(int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig, const BasisTab& tab,
                             cudaStream_t s)
{
    if constexpr (!is_tile_order(n, MIXED)) return cudaErrorInvalidValue;
    else if constexpr (MIXED) return FP_CAT(digits_mixed_, FP_N)(E, coords, boxes, dig, tab, s);
    else return digits_form<n, false>(E, coords, boxes, dig, tab, s);
}

template <int n, bool MIXED>
static int64_t digits_bytes_if()
{
    if constexpr (is_tile_order(n, MIXED)) return TileBytes<n, MIXED>::v;
    else return 0;
}

cudaError_t FP_CAT(solve_order_, FP_N)(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp,
                                       int block, cudaStream_t s)
{
    return solve_n<FP_N>(a, npairs, tab, fp, block, s);
}

cudaError_t FP_CAT(newton_order_, FP_N)(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp,
                                        int block, unsigned grid, cudaStream_t s)
{
    return newton_n<FP_N>(a, npairs, tab, fp, block, grid, s);
}

int FP_CAT(newton_fit_order_, FP_N)(bool mixed, int block) { return newton_fit<FP_N>(mixed, block); }

cudaError_t FP_CAT(digits_order_, FP_N)(bool mixed, int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig,
                                        const BasisTab& tab, cudaStream_t s)
{
    return mixed ? digits_if<FP_N, true>(E, coords, boxes, dig, tab, s)
                 : digits_if<FP_N, false>(E, coords, boxes, dig, tab, s);
}

int64_t FP_CAT(digits_bytes_order_, FP_N)(bool mixed)
{
    return mixed ? digits_bytes_if<FP_N, true>() : digits_bytes_if<FP_N, false>();
}

}  // namespace fpg
