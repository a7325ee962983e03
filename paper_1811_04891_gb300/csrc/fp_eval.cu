// fp_eval.cu -- findpts_eval (Sec. 2.1): interpolate F nodal fields at located
// points by sum factorisation, out[f][p] = sum_ijk F_ijk h_i(r) h_j(s) h_k(t),
// in FP64; quiet NaN for points that were not found.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "fp_common.cuh"
#include "fp_internal.h"

namespace fpg {

// ---------------------------------------------------------------------------
// Evaluation by planes: the n planes k of a point's element are contracted by
// n neighbouring lanes, then one lane per field adds them up over k.  Every
// value takes the operations of the one-thread form (contract, contract_df)
// in the same order, so the two agree bit for bit.
//
// Up to some 10^5 values the one-thread form leaves the GPU nearly empty: its
// time is that of one thread's chain of n^3 terms per field, with every load
// a row of its own.  By planes the chain is n times shorter and a warp works
// on few elements at a time.  The basis is evaluated once per group, one
// direction a lane (one FP64 basis a warp instead of three).
// ---------------------------------------------------------------------------
template <int n> constexpr int kPlaneGroup = n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16;   // lanes of a point

struct PlanesDf {                       // posted fields
    using W = float2;                   // weights and plane sums: float pairs
    using V = float2;
    static __device__ __forceinline__ W weight(double h)
    {
        const df a = df_split(h);
        return make_float2(a.hi, a.lo);
    }
    template <int n>
    static __device__ __forceinline__ W plane(const V* __restrict__ F, const W* __restrict__ w)
    {
        float rh[n], rl[n];
#pragma unroll
        for (int i = 0; i < n; ++i) {
            rh[i] = w[i].x;
            rl[i] = w[i].y;
        }
        df c = {0.0f, 0.0f};
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            const W s = w[n + j];
            df_fma_acc(c, row_df<n>(F + n * j, rh, rl), s.x, s.y);
        }
        df_norm(c);
        return make_float2(c.hi, c.lo);
    }
    template <int n>
    static __device__ __forceinline__ double sum(const W* __restrict__ c, const W* __restrict__ t)
    {
        df acc = {0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < n; ++k) df_fma_acc(acc, df{c[k].x, c[k].y}, t[k].x, t[k].y);
        return (double)acc.hi + (double)acc.lo;
    }
};

struct PlanesF64 {
    using W = double;
    using V = double;
    static __device__ __forceinline__ W weight(double h) { return h; }
    template <int n>
    static __device__ __forceinline__ W plane(const V* __restrict__ F, const W* __restrict__ w)
    {
        double hr[n];
#pragma unroll
        for (int i = 0; i < n; ++i) hr[i] = w[i];
        double c = 0.0;
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            double v[n];
            load_row<n>(F + n * j, v);
            double u = 0.0;
#pragma unroll
            for (int i = 0; i < n; ++i) u = fma(hr[i], v[i], u);
            c = fma(w[n + j], u, c);
        }
        return c;
    }
    template <int n>
    static __device__ __forceinline__ double sum(const W* __restrict__ c, const W* __restrict__ t)
    {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < n; ++k) acc = fma(t[k], c[k], acc);
        return acc;
    }
};

template <int n, class O>
struct PlaneSm {
    static constexpr int G = kPlaneGroup<n>;
    typename O::W w[32 / G][3 * n];     // basis values in r, s, t
    typename O::W c[32 / G][G * n];     // plane sums of up to G fields
};

// the basis values at (r0, r1, r2) = R(0), R(1), R(2)
template <int n, class O, class R>
__device__ __forceinline__ void plane_basis(typename O::W* w, int g, const BasisTab& tab, R&& r)
{
    for (int d = g; d < 3; d += kPlaneGroup<n>) {
        double h[n];
        lagrange_h<n, double>(tab.xi, tab.ci, r(d), h);
#pragma unroll
        for (int i = 0; i < n; ++i) w[d * n + i] = O::weight(h[i]);
    }
}

// the F fields at a group's point (w set); every lane of the warp takes part
template <int n, class O>
__device__ __forceinline__ void plane_values(const typename O::W* w, typename O::W* c, int g, bool ok,
                                             const typename O::V* __restrict__ fields, int64_t E, int F, int e,
                                             double* __restrict__ out, int64_t P, int64_t p)
{
    constexpr int G = kPlaneGroup<n>, n2 = n * n;
    for (int f0 = 0; f0 < F; f0 += G) {
        const int nf = min(G, F - f0);
        __syncwarp();
        if (ok && g < n)
            for (int f = 0; f < nf; ++f)
                c[f * n + g] = O::template plane<n>(fields + (((int64_t)(f0 + f) * E + e) * n + g) * n2, w);
        __syncwarp();
        if (ok && g < nf) out[(int64_t)(f0 + g) * P + p] = O::template sum<n>(c + g * n, w + 2 * n);
    }
}

// points in the caller's order (k_eval, k_eval_df), or posted points (basis
// and pe: k_eval_points_df)
template <int n, class O>
__global__ void __launch_bounds__(128) k_eval_planes(int64_t E, int64_t P, const int32_t* __restrict__ code,
                                                     const int32_t* __restrict__ elem, const double* __restrict__ rst,
                                                     const float* __restrict__ basis, int F,
                                                     const typename O::V* __restrict__ fields, double* __restrict__ out,
                                                     BasisTab tab)
{
    constexpr int G = kPlaneGroup<n>;
    __shared__ PlaneSm<n, O> sm[4];
    PlaneSm<n, O>& S = sm[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, g = lane % G, gr = lane / G;
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    const int e = p < P ? elem[p] : -1;
    const bool ok = e >= 0 && e < E && (!code || (code[p] != FP_CODE_NOT_FOUND && code[p] != FP_CODE_RETRY));
    typename O::W* w = S.w[gr];
    if (ok) {
        if constexpr (sizeof(typename O::V) == sizeof(float2) && !std::is_same_v<O, PlanesF64>) {
            if (basis) {
                for (int i = g; i < n; i += G)
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        w[d * n + i] = make_float2(__ldg(basis + ((int64_t)(2 * d) * n + i) * P + p),
                                                   __ldg(basis + ((int64_t)(2 * d + 1) * n + i) * P + p));
            } else {
                plane_basis<n, O>(w, g, tab, [&](int d) { return rst[d * P + p]; });
            }
        } else {
            plane_basis<n, O>(w, g, tab, [&](int d) { return rst[d * P + p]; });
        }
    } else if (p < P) {
        for (int f = g; f < F; f += G) out[(int64_t)f * P + p] = __longlong_as_double(0x7ff8000000000000ULL);
    }
    plane_values<n, O>(w, S.c[gr], g, ok, fields, E, F, e, out, P, p);
}

struct EvalPairsArgs {
    int64_t E, P, cap;
    const int32_t* dcount;
    const int32_t* order;
    const int32_t* pair_elem;
    const int32_t* pair_pt;
    const double* prst;
    EvalSpec ev;
    const int32_t* s_lo;      // batch groups: the group's sorted positions [*s_lo, *s_hi)
    const int32_t* s_hi;
    int32_t ebase;            // batch groups: subtracted from pair_elem
    int walk;                 // pair results at sorted positions (else at pair slots)
};

// winning pairs in the find's element-sorted order (k_eval_pairs)
template <int n, class O>
__global__ void __launch_bounds__(128) k_eval_pairs_planes(EvalPairsArgs A, const typename O::V* __restrict__ fields,
                                                           BasisTab tab)
{
    constexpr int G = kPlaneGroup<n>;
    __shared__ PlaneSm<n, O> sm[4];
    PlaneSm<n, O>& S = sm[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, g = lane % G, gr = lane / G;
    const int64_t t = *A.dcount, s1 = t < A.cap ? t : A.cap;
    const int64_t step = (int64_t)gridDim.x * 4 * (32 / G);
    for (int64_t base = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * (32 / G); base < s1; base += step) {
        const int64_t s = base + gr;
        int32_t p = -1;
        int e = 0;
        if (s < s1) {
            const int32_t q = A.order[s];
            p = A.pair_pt[q];
            if (p >= 0) {                                 // the point's winning pair
                e = A.pair_elem[q];
                const int64_t w = A.walk ? s : q;
                plane_basis<n, O>(S.w[gr], g, tab, [&](int d) { return A.prst[d * A.cap + w]; });
            }
        }
        plane_values<n, O>(S.w[gr], S.c[gr], g, p >= 0, fields, A.E, A.ev.F, e, A.ev.out, A.P, p);
        __syncwarp();                                     // the next pairs overwrite the basis
    }
}

struct EvalArgs {
    int64_t E;
    int64_t P;
    const int32_t* code;
    const int32_t* elem;
    const double* rst;
    int F;
    const double* fields;
    double* out;
};

// One thread per point, or (SPLIT) one thread per (point, field): small
// calls (an interface sub-iteration evaluates a few 10^4 points) are
// latency-bound, and splitting the fields gives F times the threads; each
// field's operations are the same either way.
template <int n, bool SPLIT>
__global__ void __launch_bounds__(128) k_eval(EvalArgs A, BasisTab tab)
{
    constexpr int n3 = n * n * n;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t p = SPLIT ? t / A.F : t;
    if (p >= A.P) return;
    const int f0 = SPLIT ? (int)(t % A.F) : 0, f1 = SPLIT ? f0 + 1 : A.F;
    const int e = A.elem[p];
    if (A.code[p] == FP_CODE_NOT_FOUND || e < 0 || e >= A.E) {
        for (int f = f0; f < f1; ++f) A.out[(int64_t)f * A.P + p] = __longlong_as_double(0x7ff8000000000000ULL);
        return;
    }
    double hr[n], hs[n], ht[n];
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[p], hr);
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[A.P + p], hs);
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[2 * A.P + p], ht);
    for (int f = f0; f < f1; ++f)
        A.out[(int64_t)f * A.P + p] = contract<n, double>(A.fields + ((int64_t)f * A.E + e) * n3, hr, hs, ht);
}

// calls with at most this many (point, field) values take one thread each
constexpr int64_t kSplitEval = int64_t(1) << 21;

// Which calls evaluate by planes.  A group takes its point's fields one after
// the other, and the groups of n >= 9 leave up to 7 of 16 lanes idle, so it is
// for few values of few fields (more of them where the chain of one thread is
// long).  us, one thread per value / planes, points of one element side by
// side (points in any order gain more, up to twice as much):
//   FP64    n = 3    F = 3: 2,000 points 6/5;  F = 6: 2,000 6/7
//           n = 8    F = 1: 2,000 points 34/7, 10,000 34/21, 20,000 47/37;  F = 6: 2,000 36/25;  F = 12: 500 37/46
//           n = 10   F = 1: 5,000 54/29, 10,000 55/51;  F = 3: 5,000 57/64;  F = 6: 2,000 58/49;  F = 12: 500 59/64
//           n = 13   F = 6: 2,000 121/78;  F = 12: 500 158/113
//   posted  n = 8    F = 1: 2,000 24/8, 20,000 32/29;  F = 3: 5,000 27/27;  F = 12: 500 32/42
//           n = 10   F = 3: 5,000 44/37;  F = 6: 2,000 47/35;  F = 12: 500 65/54
static bool eval_by_planes(int n, int64_t P, int F, bool df)
{
    const int fields = n <= 3 ? 4 : n <= 9 || (n == 10 && !df) ? 6 : 12;
    return F <= fields && P * F <= (n <= 8 ? 20000 : df ? 15000 : 12000);
}

// Posted points in thread form share their rows' loads (see
// k_eval_points_df).  us, thread / planes, points of one element side by side:
//   n = 6    F = 1: 2,000 points 10/4, 20,000 11/8;  F = 3: 5,000 11/7;  F = 6: 500 10/10
//   n = 8    F = 1: 2,000 17/5, 10,000 18/13, 20,000 18/22;  F = 3: 2,000 17/12, 5,000 18/21;  F = 6: 500 17/21
//   n = 10   F = 1: 2,000 36/7, 20,000 38/33;  F = 3: 5,000 37/27;  F = 6: 2,000 37/29
//   n = 13   F = 1: 2,000 69/15, 20,000 75/69;  F = 6: 2,000 72/79 (in any order 141/92)
static bool points_by_planes(int n, int64_t P, int F)
{
    return F <= (n <= 9 ? 3 : 6) && P * F <= (n == 8 ? 10000 : 20000);
}

// Sorted pairs of a find (thread / planes / one thread per pair and field, us):
//   FP64    n = 6    F = 3: 20,000 points 60/49/48, 65,000 114/147/127
//           n = 8    F = 3: 20,000 126/79/94, 40,000 185/148/172, 65,000 246/241/258
//           n = 10   F = 1: 5,000 59/30/59, 20,000 84/101/84;  F = 6: 2,000 332/49/64, 5,000 321/117/86, 65,000 868/1287/857
//   posted  n = 6    F = 3: 20,000 38/24/34, 40,000 46/39/50, 65,000 55/59/71
//           n = 7    F = 3: 40,000 82/58/71, 65,000 93/81/94;  F = 6: 65,000 161/149/157
//           n = 8    F = 3: 10,000 104/42/52, 20,000 102/72/65, 40,000 115/122/90, 65,000 123/193/114;  F = 12: 5,000 512/86/78
//           n = 13   F = 6: 2,000 408/146/99, 20,000 385/500/226, 65,000 631/1335/550
// The basis of every field costs more than the threads give once the pairs
// fill the GPU several times, sooner the lower the order.
enum PairForm { PAIR_THREAD, PAIR_PLANES, PAIR_FIELD };
constexpr int kFieldMinN = 7;

static PairForm pair_form(int n, int64_t P, int F, bool df)
{
    if (n >= 9 ? P * F <= (df ? 10000 : n >= 12 ? 15000 : 12000) : P <= 20000 && !(df && n == 8 && P * F > 30000))
        return PAIR_PLANES;
    return n >= kFieldMinN && F <= 16 && P <= (df || n >= 9 ? 65536 : 50000) ? PAIR_FIELD : PAIR_THREAD;
}

template <int n>
static unsigned plane_grid(int64_t count)
{
    return (unsigned)((count * kPlaneGroup<n> + 127) / 128);
}

cudaError_t launch_eval(int n, int64_t E, int64_t P, const int32_t* code, const int32_t* elem, const double* rst,
                        int F, const double* fields, double* out, const BasisTab& tab, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    EvalArgs a{E, P, code, elem, rst, F, fields, out};
    const bool split = P * F <= kSplitEval, planes = eval_by_planes(n, P, F, false);
    const unsigned grid = (unsigned)(((split ? P * F : P) + 127) / 128);
    switch (n) {
#define FP_CASE(NN)                                                                                           \
    case NN:                                                                                                  \
        if (planes) k_eval_planes<NN, PlanesF64><<<plane_grid<NN>(P), 128, 0, s>>>(E, P, code, elem, rst, nullptr, F, fields, out, tab); \
        else if (split) k_eval<NN, true><<<grid, 128, 0, s>>>(a, tab);                                        \
        else k_eval<NN, false><<<grid, 128, 0, s>>>(a, tab);                                                  \
        break;
        FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9)
        FP_CASE(10) FP_CASE(11) FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace fpg

// ---------------------------------------------------------------------------
// Double-float evaluation for the mixed form.
//
// Every nodal value f is posted once as an unevaluated sum of two floats,
// f = f_hi + f_lo (f_hi = fl(f), f_lo = fl(f - f_hi), 48 significant bits),
// and each basis value h(r), computed in FP64, is split the same way.  The
// contraction then runs on the FP32 pipes: each product f*h is formed exactly
// in its leading part (p = f_hi*h_hi, e = fma(f_hi, h_hi, -p)) plus the
// first-order cross terms, and the sum is carried as a (hi, lo) pair with an
// error-free two-sum.  The result is rounded to FP64 at the end.  Relative
// error is a few units of 2^-48 times the sum of |terms|.
// ---------------------------------------------------------------------------
namespace fpg {

struct Eval2Args {
    int64_t E;
    int64_t P;
    const int32_t* code;
    const int32_t* elem;
    const double* rst;
    int F;
    const float2* fields;     // [F][E][n3] posted: per row n high parts, then n low parts
    double* out;
};

template <int n, bool SPLIT>
__global__ void __launch_bounds__(128) k_eval_df(Eval2Args A, BasisTab tab)
{
    constexpr int n3 = n * n * n;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t p = SPLIT ? t / A.F : t;
    if (p >= A.P) return;
    const int f0 = SPLIT ? (int)(t % A.F) : 0, f1 = SPLIT ? f0 + 1 : A.F;
    const int e = A.elem[p];
    if (A.code[p] == FP_CODE_NOT_FOUND || A.code[p] == FP_CODE_RETRY || e < 0 || e >= A.E) {
        for (int f = f0; f < f1; ++f) A.out[(int64_t)f * A.P + p] = __longlong_as_double(0x7ff8000000000000ULL);
        return;
    }
    double hr[n], hs[n], ht[n];
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[p], hr);
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[A.P + p], hs);
    lagrange_h<n, double>(tab.xi, tab.ci, A.rst[2 * A.P + p], ht);
    float rh[n], rl[n], sh[n], sl[n], th[n], tl[n];
#pragma unroll
    for (int i = 0; i < n; ++i) {
        df a = df_split(hr[i]), b = df_split(hs[i]), c = df_split(ht[i]);
        rh[i] = a.hi; rl[i] = a.lo; sh[i] = b.hi; sl[i] = b.lo; th[i] = c.hi; tl[i] = c.lo;
    }
    for (int f = f0; f < f1; ++f)
        A.out[(int64_t)f * A.P + p] = contract_df<n>(A.fields + ((int64_t)f * A.E + e) * n3, rh, rl, sh, sl, th, tl);
}

// ---- posted points: the split basis values of located points, computed once
// and reused by every evaluation at the same (e, r) (the interface points of
// a Schwarz step are evaluated once per sub-iteration).  Layout [6n][P]:
// rh, rl, sh, sl, th, tl, each n rows, so consecutive threads load
// consecutive words; elem = -1 marks points without a value.
template <int n>
__global__ void k_points_basis(int64_t P, const int32_t* __restrict__ code, const int32_t* __restrict__ elem,
                               const double* __restrict__ rst, float* __restrict__ basis, int32_t* __restrict__ pe,
                               BasisTab tab)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= P) return;
    const bool ok = !(code[p] == FP_CODE_NOT_FOUND || code[p] == FP_CODE_RETRY || elem[p] < 0);
    pe[p] = ok ? elem[p] : -1;
    if (!ok) return;
    double h[n];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        lagrange_h<n, double>(tab.xi, tab.ci, rst[d * P + p], h);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const df v = df_split(h[i]);
            basis[((int64_t)(2 * d) * n + i) * P + p] = v.hi;
            basis[((int64_t)(2 * d + 1) * n + i) * P + p] = v.lo;
        }
    }
}

// One thread per (point, field).  A block takes one field at consecutive
// points: interface nodes follow the faces, so these lie in one element, and
// the lanes of a warp load the same row in one access instead of one per
// field.  32,768 interface nodes, 4 fields, N = 7: 71 -> 49 us.
__host__ __device__ __forceinline__ unsigned value_blocks(int64_t P) { return (unsigned)((P + 127) / 128); }

template <int n>
__global__ void __launch_bounds__(128) k_eval_points_df(int64_t E, int64_t P, int F, const int32_t* __restrict__ pe,
                                                        const float* __restrict__ basis,
                                                        const float2* __restrict__ fields, double* __restrict__ out)
{
    constexpr int n3 = n * n * n;
    const unsigned nb = value_blocks(P);
    const int f = (int)(blockIdx.x / nb);
    const int64_t p = (int64_t)(blockIdx.x - f * nb) * blockDim.x + threadIdx.x;
    if (p >= P) return;
    const int e = pe[p];
    if (e < 0 || e >= E) {
        out[(int64_t)f * P + p] = __longlong_as_double(0x7ff8000000000000ULL);
        return;
    }
    float rh[n], rl[n], sh[n], sl[n], th[n], tl[n];
#pragma unroll
    for (int i = 0; i < n; ++i) {
        rh[i] = __ldg(basis + (int64_t)(0 * n + i) * P + p);
        rl[i] = __ldg(basis + (int64_t)(1 * n + i) * P + p);
        sh[i] = __ldg(basis + (int64_t)(2 * n + i) * P + p);
        sl[i] = __ldg(basis + (int64_t)(3 * n + i) * P + p);
        th[i] = __ldg(basis + (int64_t)(4 * n + i) * P + p);
        tl[i] = __ldg(basis + (int64_t)(5 * n + i) * P + p);
    }
    out[(int64_t)f * P + p] = contract_df<n>(fields + ((int64_t)f * E + e) * n3, rh, rl, sh, sl, th, tl);
}

// posted fields: value v -> (hi, lo) = (fl32(v), fl32(v - hi)), each row of
// n nodes stored as its n high parts then its n low parts (see row_df)
__global__ void k_split_df(int64_t count, int n, const double* __restrict__ src, float2* __restrict__ dst)
{
    float* d = reinterpret_cast<float*>(dst);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / n, c = i - row * n;
        const double v = src[i];
        const float h = (float)v;
        d[2 * n * row + c] = h;
        d[2 * n * row + n + c] = (float)(v - (double)h);
    }
}

cudaError_t launch_split_df(int64_t count, int n, const double* src, float2* dst, cudaStream_t s)
{
    const int64_t blocks = std::min<int64_t>((count + 255) / 256, 152 * 32);
    k_split_df<<<(unsigned)std::max<int64_t>(blocks, 1), 256, 0, s>>>(count, n, src, dst);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_points_basis(int n, int64_t P, const int32_t* code, const int32_t* elem, const double* rst,
                                float* basis, int32_t* pe, const BasisTab& tab, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((P + 127) / 128);
    switch (n) {
#define FP_CASE(NN) \
    case NN: k_points_basis<NN><<<grid, 128, 0, s>>>(P, code, elem, rst, basis, pe, tab); break;
        FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9)
        FP_CASE(10) FP_CASE(11) FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_eval_points_df(int n, int64_t E, int64_t P, int F, const int32_t* pe, const float* basis,
                                  const float2* fields, double* out, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    const unsigned grid = value_blocks(P) * F;
    const bool planes = points_by_planes(n, P, F);
    switch (n) {
#define FP_CASE(NN)                                                                                           \
    case NN:                                                                                                  \
        if (planes) k_eval_planes<NN, PlanesDf><<<plane_grid<NN>(P), 128, 0, s>>>(E, P, nullptr, pe, nullptr, basis, F, fields, out, BasisTab()); \
        else k_eval_points_df<NN><<<grid, 128, 0, s>>>(E, P, F, pe, basis, fields, out);                      \
        break;
        FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9)
        FP_CASE(10) FP_CASE(11) FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_eval_df(int n, int64_t E, int64_t P, const int32_t* code, const int32_t* elem, const double* rst,
                           int F, const float2* fields, double* out, const BasisTab& tab, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    Eval2Args a{E, P, code, elem, rst, F, fields, out};
    const bool split = P * F <= kSplitEval, planes = eval_by_planes(n, P, F, true);
    const unsigned grid = (unsigned)(((split ? P * F : P) + 127) / 128);
    switch (n) {
#define FP_CASE(NN)                                                     \
    case NN:                                                            \
        if (planes) k_eval_planes<NN, PlanesDf><<<plane_grid<NN>(P), 128, 0, s>>>(E, P, code, elem, rst, nullptr, F, fields, out, tab); \
        else if (split) k_eval_df<NN, true><<<grid, 128, 0, s>>>(a, tab);    \
        else k_eval_df<NN, false><<<grid, 128, 0, s>>>(a, tab);         \
        break;
        FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9)
        FP_CASE(10) FP_CASE(11) FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace fpg

// ---------------------------------------------------------------------------
// Fused evaluation in the element-sorted pair order of the find (one thread
// per winning pair; neighbouring threads work on the same element, so its
// field rows are served from L1 instead of being re-read from DRAM).
// ---------------------------------------------------------------------------
namespace fpg {

template <int n>
__device__ __forceinline__ void eval_point_f64(const double* __restrict__ F64, int64_t E, int F, int e, double r0,
                                               double r1, double r2, const BasisTab& tab, double* __restrict__ out,
                                               int64_t P, int64_t p)
{
    constexpr int n3 = n * n * n;
    double hr[n], hs[n], ht[n];
    lagrange_h<n, double>(tab.xi, tab.ci, r0, hr);
    lagrange_h<n, double>(tab.xi, tab.ci, r1, hs);
    lagrange_h<n, double>(tab.xi, tab.ci, r2, ht);
    for (int f = 0; f < F; ++f)
        out[(int64_t)f * P + p] = contract<n, double>(F64 + ((int64_t)f * E + e) * n3, hr, hs, ht);
}

template <int n>
__device__ __forceinline__ void eval_point_df(const float2* __restrict__ Fdf, int64_t E, int F, int e, double r0,
                                              double r1, double r2, const BasisTab& tab, double* __restrict__ out,
                                              int64_t P, int64_t p)
{
    constexpr int n3 = n * n * n;
    double hr[n], hs[n], ht[n];
    lagrange_h<n, double>(tab.xi, tab.ci, r0, hr);
    lagrange_h<n, double>(tab.xi, tab.ci, r1, hs);
    lagrange_h<n, double>(tab.xi, tab.ci, r2, ht);
    float rh[n], rl[n], sh[n], sl[n], th[n], tl[n];
#pragma unroll
    for (int i = 0; i < n; ++i) {
        df a = df_split(hr[i]), b = df_split(hs[i]), c = df_split(ht[i]);
        rh[i] = a.hi; rl[i] = a.lo; sh[i] = b.hi; sl[i] = b.lo; th[i] = c.hi; tl[i] = c.lo;
    }
    for (int f = 0; f < F; ++f)
        out[(int64_t)f * P + p] = contract_df<n>(Fdf + ((int64_t)f * E + e) * n3, rh, rl, sh, sl, th, tl);
}


// one thread per winning pair, or (FIELD, gridDim.y = F) one per pair and
// field; a kernel of its own each, which leaves the compiler its registers
// (n = 8, posted, F = 3, 65,000 pairs 103 us, 123 in one)
template <int n, bool DF, bool FIELD>
__global__ void __launch_bounds__(128) k_eval_pairs(EvalPairsArgs A, BasisTab tab)
{
    constexpr int n3 = n * n * n;
    const int nf = FIELD ? A.ev.F / (int)gridDim.y : 0;   // (1; a constant 1 gives slower code)
    const int64_t f0 = (int64_t)blockIdx.y * nf;
    int64_t s0 = 0, s1;
    if (A.s_lo) {
        s0 = *A.s_lo;
        s1 = *A.s_hi;
    } else {
        const int64_t t = *A.dcount;
        s1 = t < A.cap ? t : A.cap;
    }
    for (int64_t s = s0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < s1; s += (int64_t)gridDim.x * blockDim.x) {
        const int32_t q = A.order[s];
        const int32_t p = A.pair_pt[q];
        if (p < 0) continue;                              // not the point's winning pair
        const int e = A.pair_elem[q] - A.ebase;
        const int64_t w = A.walk ? s : q;
        const double r0 = A.prst[w], r1 = A.prst[A.cap + w], r2 = A.prst[2 * A.cap + w];
        if constexpr (FIELD) {
            if (DF) eval_point_df<n>(A.ev.fdf + f0 * A.E * n3, A.E, nf, e, r0, r1, r2, tab, A.ev.out + f0 * A.P, A.P, p);
            else eval_point_f64<n>(A.ev.f64 + f0 * A.E * n3, A.E, nf, e, r0, r1, r2, tab, A.ev.out + f0 * A.P, A.P, p);
        } else {
            if (DF) eval_point_df<n>(A.ev.fdf, A.E, A.ev.F, e, r0, r1, r2, tab, A.ev.out, A.P, p);
            else eval_point_f64<n>(A.ev.f64, A.E, A.ev.F, e, r0, r1, r2, tab, A.ev.out, A.P, p);
        }
    }
}

// Fused double-float evaluation with each element's posted fields staged in
// shared memory: a block takes kStageTile consecutive sorted pairs (the pairs
// of one element are consecutive), copies the fields of each element the
// tile touches into shared memory once, in ascending element order, and the
// threads whose pairs lie in that element read their rows from there.
constexpr int kStageTile = 128;

template <int n>
__global__ void __launch_bounds__(kStageTile) k_eval_pairs_staged(EvalPairsArgs A, BasisTab tab)
{
    constexpr int n3 = n * n * n;
    extern __shared__ float4 stage4[];               // F * n3 float2: the current element's fields
    float2* stage = reinterpret_cast<float2*>(stage4);
    __shared__ int ecur;
    int64_t s0 = 0, s1;
    if (A.s_lo) {
        s0 = *A.s_lo;
        s1 = *A.s_hi;
    } else {
        const int64_t t = *A.dcount;
        s1 = t < A.cap ? t : A.cap;
    }
    const int F = A.ev.F;
    for (int64_t base = s0 + (int64_t)blockIdx.x * kStageTile; base < s1;
         base += (int64_t)gridDim.x * kStageTile) {
        const int64_t s = base + threadIdx.x;
        int32_t p = -1;
        int e = -1;
        float rh[n], rl[n], sh[n], sl[n], th[n], tl[n];
        if (s < s1) {
            const int32_t q = A.order[s];
            p = A.pair_pt[q];
            e = A.pair_elem[q] - A.ebase;
            if (p >= 0) {
                const int64_t w = A.walk ? s : q;
                double hr[n], hs[n], ht[n];
                lagrange_h<n, double>(tab.xi, tab.ci, A.prst[w], hr);
                lagrange_h<n, double>(tab.xi, tab.ci, A.prst[A.cap + w], hs);
                lagrange_h<n, double>(tab.xi, tab.ci, A.prst[2 * A.cap + w], ht);
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const df a = df_split(hr[i]), b = df_split(hs[i]), c = df_split(ht[i]);
                    rh[i] = a.hi; rl[i] = a.lo; sh[i] = b.hi; sl[i] = b.lo; th[i] = c.hi; tl[i] = c.lo;
                }
            }
        }
        bool done = p < 0;                           // losers and threads past the end have nothing to do
        for (;;) {
            if (threadIdx.x == 0) ecur = INT_MAX;
            __syncthreads();
            if (!done) atomicMin(&ecur, e);
            __syncthreads();
            const int ec = ecur;
            if (ec == INT_MAX) break;                // uniform: every thread read the same value
            for (int f = 0; f < F; ++f) {
                const float2* src = A.ev.fdf + ((int64_t)f * A.E + ec) * n3;
                if constexpr (n3 % 2 == 0) {
                    const float4* s4 = reinterpret_cast<const float4*>(src);
                    float4* d4 = stage4 + f * (n3 / 2);
                    for (int v = threadIdx.x; v < n3 / 2; v += kStageTile) d4[v] = __ldg(s4 + v);
                } else {
                    for (int v = threadIdx.x; v < n3; v += kStageTile) stage[f * n3 + v] = __ldg(src + v);
                }
            }
            __syncthreads();
            if (!done && e == ec) {
                for (int f = 0; f < F; ++f)
                    A.ev.out[(int64_t)f * A.P + p] = contract_df<n, true>(stage + f * n3, rh, rl, sh, sl, th, tl);
                done = true;
            }
            __syncthreads();                         // the next element overwrites the stage
        }
    }
}

// staging is used when one element's posted fields fit in this much shared
// memory (larger ones are evaluated from L1 / L2 as without staging)
constexpr int64_t kStageMaxBytes = 48 * 1024;

cudaError_t launch_eval_pairs(int n, int64_t E, int64_t P, const int32_t* dcount, int64_t cap, const int32_t* order,
                              const int32_t* pair_elem, const int32_t* pair_pt, const double* prst,
                              const EvalSpec& ev, const BasisTab& tab, unsigned grid, cudaStream_t s,
                              const int32_t* s_lo, const int32_t* s_hi, int32_t ebase, bool walk)
{
    EvalPairsArgs a{E, P, cap, dcount, order, pair_elem, pair_pt, prst, ev, s_lo, s_hi, ebase, walk ? 1 : 0};
    const bool df = ev.fdf != nullptr;
    const int64_t stage_bytes = (int64_t)ev.F * n * n * n * (int64_t)sizeof(float2);
    const bool staged = df && ev.staged && stage_bytes <= kStageMaxBytes;
    // (batches: one thread per pair; the staging that a caller asked for comes first)
    const PairForm form = s_lo || staged ? PAIR_THREAD : pair_form(n, P, ev.F, df);
    const bool planes = form == PAIR_PLANES;
    const bool field = form == PAIR_FIELD;
    const dim3 grid2(grid, ev.F);
    switch (n) {
#define FP_CASE(NN)                                                                       \
    case NN:                                                                              \
        if (planes && df) k_eval_pairs_planes<NN, PlanesDf><<<grid * kPlaneGroup<NN>, 128, 0, s>>>(a, ev.fdf, tab); \
        else if (planes) k_eval_pairs_planes<NN, PlanesF64><<<grid * kPlaneGroup<NN>, 128, 0, s>>>(a, ev.f64, tab); \
        else if (staged) k_eval_pairs_staged<NN><<<grid, kStageTile, stage_bytes, s>>>(a, tab); \
        else if (field && df) k_eval_pairs<NN, true, (NN >= kFieldMinN)><<<grid2, 128, 0, s>>>(a, tab); \
        else if (field) k_eval_pairs<NN, false, (NN >= kFieldMinN)><<<grid2, 128, 0, s>>>(a, tab); \
        else if (df) k_eval_pairs<NN, true, false><<<grid, 128, 0, s>>>(a, tab);          \
        else k_eval_pairs<NN, false, false><<<grid, 128, 0, s>>>(a, tab);                 \
        break;
        FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9)
        FP_CASE(10) FP_CASE(11) FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace fpg
