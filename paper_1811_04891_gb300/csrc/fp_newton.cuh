// fp_newton.cuh -- the box-constrained trust-region Newton solver of a
// (point, candidate element) pair (Sec. 2.1) and its building blocks, shared
// by the thread-per-pair kernels (fp_solve.cu) and the tensor-core tile
// kernels (fp_tile.cuh).
#pragma once
#include "fp_common.cuh"
#include "fp_internal.h"

namespace fpg {

// number of pairs to process: the device-side total, capped by the capacity
__device__ __forceinline__ int64_t live_pairs(const int32_t* __restrict__ dcount, int64_t cap)
{
    const int64_t t = *dcount;
    return t < cap ? t : cap;
}

// ---------------------------------------------------------------------------
// Newton machinery
// ---------------------------------------------------------------------------
template <typename T>
struct ElemPtr {
    const T* X0;
    const T* X1;
    const T* X2;
};

template <int n, typename T>
__device__ __forceinline__ void eval_fJ(const ElemPtr<T>& el, const BasisTab& tab, const T (&r)[3],
                                        const T (&xs)[3], T (&f)[3], T (&J)[9])
{
    T hr[n], dr[n], hs[n], ds[n], ht[n], dt[n];
    lagrange_hd<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[0], hr, dr);
    lagrange_hd<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[1], hs, ds);
    lagrange_hd<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[2], ht, dt);
    T x[3];
    map_jac<n, T>(el.X0, el.X1, el.X2, hr, dr, hs, ds, ht, dt, x, J);
#pragma unroll
    for (int a = 0; a < 3; ++a) f[a] = x[a] - xs[a];
}

template <int n, typename T>
__device__ __forceinline__ void eval_f(const ElemPtr<T>& el, const BasisTab& tab, const T (&r)[3],
                                       const T (&xs)[3], T (&f)[3])
{
    T hr[n], hs[n], ht[n];
    lagrange_h<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[0], hr);
    lagrange_h<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[1], hs);
    lagrange_h<n, T>(Tab<T>::xi(tab), Tab<T>::ci(tab), r[2], ht);
    f[0] = contract<n, T>(el.X0, hr, hs, ht) - xs[0];
    f[1] = contract<n, T>(el.X1, hr, hs, ht) - xs[1];
    f[2] = contract<n, T>(el.X2, hr, hs, ht) - xs[2];
}

// J d = -f by cofactors; returns false when J is singular.
template <typename T>
__device__ __forceinline__ bool newton_solve3(const T (&J)[9], const T (&f)[3], T (&d)[3])
{
    const T C00 = J[4] * J[8] - J[5] * J[7], C01 = J[5] * J[6] - J[3] * J[8], C02 = J[3] * J[7] - J[4] * J[6];
    const T det = J[0] * C00 + J[1] * C01 + J[2] * C02;
    if (det == T(0) || !isfinite(det)) return false;
    const T C10 = J[2] * J[7] - J[1] * J[8], C11 = J[0] * J[8] - J[2] * J[6], C12 = J[1] * J[6] - J[0] * J[7];
    const T C20 = J[1] * J[5] - J[2] * J[4], C21 = J[2] * J[3] - J[0] * J[5], C22 = J[0] * J[4] - J[1] * J[3];
    const T id = T(1) / det;
    d[0] = -(C00 * f[0] + C10 * f[1] + C20 * f[2]) * id;
    d[1] = -(C01 * f[0] + C11 * f[1] + C21 * f[2]) * id;
    d[2] = -(C02 * f[0] + C12 * f[1] + C22 * f[2]) * id;
    return true;
}

// Gauss-Newton step with an active set: coordinates on a bound whose
// descent direction leaves the box are frozen; the remaining ones solve the
// reduced normal equations (the plain Newton step when all three are free).
// Returns the number of free coordinates.
template <typename T>
__device__ __forceinline__ int gn_step(const T (&J)[9], const T (&f)[3], const T (&r)[3], T (&d)[3])
{
    T g[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) g[b] = J[b] * f[0] + J[3 + b] * f[1] + J[6 + b] * f[2];
    bool act[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) act[b] = (r[b] <= T(-1) && g[b] > T(0)) || (r[b] >= T(1) && g[b] < T(0));
    int nfree = 0;
    for (int pass = 0; pass < 4; ++pass) {
        d[0] = d[1] = d[2] = T(0);
        int fi[3];
        nfree = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if (!act[b]) fi[nfree++] = b;
        if (nfree == 0) break;
        bool ok = false;
        if (nfree == 3) {
            ok = newton_solve3<T>(J, f, d);
        } else if (nfree == 2) {
            const int p = fi[0], q = fi[1];
            const T a00 = J[p] * J[p] + J[3 + p] * J[3 + p] + J[6 + p] * J[6 + p];
            const T a11 = J[q] * J[q] + J[3 + q] * J[3 + q] + J[6 + q] * J[6 + q];
            const T a01 = J[p] * J[q] + J[3 + p] * J[3 + q] + J[6 + p] * J[6 + q];
            const T det = a00 * a11 - a01 * a01;
            if (det > T(0)) {
                d[p] = (-a11 * g[p] + a01 * g[q]) / det;
                d[q] = (-a00 * g[q] + a01 * g[p]) / det;
                ok = true;
            }
        } else {
            const int p = fi[0];
            const T a00 = J[p] * J[p] + J[3 + p] * J[3 + p] + J[6 + p] * J[6 + p];
            if (a00 > T(0)) {
                d[p] = -g[p] / a00;
                ok = true;
            }
        }
        if (!ok) {                                   // singular: steepest descent
            for (int t = 0; t < nfree; ++t) d[fi[t]] = -g[fi[t]];
        }
        bool grew = false;
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if (!act[b] && ((r[b] <= T(-1) && d[b] < T(0)) || (r[b] >= T(1) && d[b] > T(0)))) {
                act[b] = true;
                grew = true;
            }
        if (!grew) break;
    }
    return nfree;
}

template <typename T> struct Lim;
template <> struct Lim<double> {
    static constexpr double quick = 1e-4;     // full Newton step size that hands over to chord steps
    static constexpr double chord = 1e-13;    // chord correction that confirms convergence
    static constexpr double stop = 1e-13;     // accepted step that ends a constrained solve
    static constexpr double rho_min = 1e-15;
};
template <> struct Lim<float> {
    static constexpr float quick = 2e-5f;
    static constexpr float chord = 0.0f;      // unused: the FP64 phase follows
    static constexpr float stop = 1e-6f;
    static constexpr float rho_min = 1e-7f;
};

// Box truncation of a step d at r: largest t <= 1 with r + t d in the box;
// the new point lands exactly on the bound it was cut at.
template <typename T>
__device__ __forceinline__ T box_step(const T (&r)[3], const T (&d)[3], T (&rn)[3])
{
    T t = T(1);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (d[b] > T(0) && r[b] + d[b] > T(1)) t = fmin(t, (T(1) - r[b]) / d[b]);
        if (d[b] < T(0) && r[b] + d[b] < T(-1)) t = fmin(t, (T(-1) - r[b]) / d[b]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        T v = r[b] + t * d[b];
        if (t < T(1)) {
            if (d[b] > T(0) && (T(1) - r[b]) / d[b] == t) v = T(1);
            if (d[b] < T(0) && (T(-1) - r[b]) / d[b] == t) v = T(-1);
        }
        rn[b] = fmin(T(1), fmax(T(-1), v));
    }
    return t;
}

// Chord iterations in FP64: value-only residuals with a fixed Jacobian J and
// the active-set step.  Converged when the next step is <= 1e-13 in every
// coordinate (r is then kept with its own residual).  Returns true on
// convergence; `res` is the residual norm at the returned r.
// Threshold of the chord check: 1e-13 in r, raised to the rounding level of a
// step where that is larger.  The residual x(r) - x* carries rounding errors
// of a few units of |x*|, which a step J^-1 f turns into ||J^-1|| times as
// much in r; on small elements far from the origin that exceeds 1e-13 and no
// step could confirm convergence.  2 eps |x*| ||J^-1||_inf bounds the noise.
__device__ __forceinline__ double chord_tol3(const double (&J)[9], const double (&xs)[3])
{
    const double C00 = J[4] * J[8] - J[5] * J[7], C01 = J[5] * J[6] - J[3] * J[8], C02 = J[3] * J[7] - J[4] * J[6];
    const double det = J[0] * C00 + J[1] * C01 + J[2] * C02;
    if (!(fabs(det) > 0.0) || !isfinite(det)) return Lim<double>::chord;
    const double C10 = J[2] * J[7] - J[1] * J[8], C11 = J[0] * J[8] - J[2] * J[6], C12 = J[1] * J[6] - J[0] * J[7];
    const double C20 = J[1] * J[5] - J[2] * J[4], C21 = J[2] * J[3] - J[0] * J[5], C22 = J[0] * J[4] - J[1] * J[3];
    const double rows = fmax(fabs(C00) + fabs(C10) + fabs(C20),
                             fmax(fabs(C01) + fabs(C11) + fabs(C21), fabs(C02) + fabs(C12) + fabs(C22)));
    const double xm = fmax(fabs(xs[0]), fmax(fabs(xs[1]), fabs(xs[2])));
    return fmax(Lim<double>::chord, 4.440892098500626e-16 * xm * rows / fabs(det));
}

// ---- one warp per pair: the n^2 rows of the contractions are split over the
// lanes, partial sums reduced to lane 0 in a fixed order and broadcast, so
// every lane holds the same bits and the Newton control flow stays uniform
// across the warp.  Used for the few pairs of the mixed form's fallback, whose
// cost is the latency of one long FP64 solve rather than throughput.
__device__ __forceinline__ double warp_sum_bcast(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);
}

template <int n>
__device__ void eval_fJ_warp(const ElemPtr<double>& el, const BasisTab& tab, const double (&r)[3],
                             const double (&xs)[3], double (&f)[3], double (&J)[9])
{
    double hr[n], dr[n], hs[n], ds[n], ht[n], dt[n];
    lagrange_hd<n, double>(tab.xi, tab.ci, r[0], hr, dr);
    lagrange_hd<n, double>(tab.xi, tab.ci, r[1], hs, ds);
    lagrange_hd<n, double>(tab.xi, tab.ci, r[2], ht, dt);
    double x[3] = {0, 0, 0}, xr[3] = {0, 0, 0}, xsd[3] = {0, 0, 0}, xt[3] = {0, 0, 0};
    const int lane = threadIdx.x & 31;
    for (int q = lane; q < n * n; q += 32) {              // row q = j + n k
        const int j = q % n, k = q / n;
        const double hsj = hs[j], dsj = ds[j], htk = ht[k], dtk = dt[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double v[n];
            load_row<n>((a == 0 ? el.X0 : (a == 1 ? el.X1 : el.X2)) + n * q, v);
            double u = 0.0, w = 0.0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                u = fma(hr[i], v[i], u);
                w = fma(dr[i], v[i], w);
            }
            x[a] = fma(htk, hsj * u, x[a]);
            xr[a] = fma(htk, hsj * w, xr[a]);
            xsd[a] = fma(htk, dsj * u, xsd[a]);
            xt[a] = fma(dtk, hsj * u, xt[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        f[a] = warp_sum_bcast(x[a]) - xs[a];
        J[3 * a + 0] = warp_sum_bcast(xr[a]);
        J[3 * a + 1] = warp_sum_bcast(xsd[a]);
        J[3 * a + 2] = warp_sum_bcast(xt[a]);
    }
}

template <int n>
__device__ void eval_f_warp(const ElemPtr<double>& el, const BasisTab& tab, const double (&r)[3],
                            const double (&xs)[3], double (&f)[3])
{
    double hr[n], hs[n], ht[n];
    lagrange_h<n, double>(tab.xi, tab.ci, r[0], hr);
    lagrange_h<n, double>(tab.xi, tab.ci, r[1], hs);
    lagrange_h<n, double>(tab.xi, tab.ci, r[2], ht);
    double x[3] = {0, 0, 0};
    const int lane = threadIdx.x & 31;
    for (int q = lane; q < n * n; q += 32) {
        const double c = ht[q / n] * hs[q % n];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double v[n];
            load_row<n>((a == 0 ? el.X0 : (a == 1 ? el.X1 : el.X2)) + n * q, v);
            double u = 0.0;
#pragma unroll
            for (int i = 0; i < n; ++i) u = fma(hr[i], v[i], u);
            x[a] = fma(c, u, x[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) f[a] = warp_sum_bcast(x[a]) - xs[a];
}

template <int n, bool WARP = false>
__device__ bool chord64(const ElemPtr<double>& el, const BasisTab& tab, const double (&xs)[3], double (&r)[3],
                        const double (&J)[9], double& res, int max_chord)
{
    const double tol = chord_tol3(J, xs);
    for (int it = 0; it < max_chord; ++it) {
        double f[3];
        if constexpr (WARP) eval_f_warp<n>(el, tab, r, xs, f);
        else eval_f<n, double>(el, tab, r, xs, f);
        res = sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
        if (!(res > 0.0)) return true;
        double d[3];
        if (gn_step<double>(J, f, r, d) == 0) return true;         // KKT point at a vertex
        double rn[3];
        box_step<double>(r, d, rn);
        const double sn = fmax(fabs(rn[0] - r[0]), fmax(fabs(rn[1] - r[1]), fabs(rn[2] - r[2])));
        if (sn <= tol) return true;
        r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
    }
    return false;
}

// Box-constrained trust-region Newton (Sec. 2.1) from r (in/out); J returns
// the Jacobian at (or one small step before) the returned r.  Returns the
// residual norm ||x(r) - x*|| at the returned r.  With FINAL (FP64) a small
// full Newton step hands over to chord iterations with the current Jacobian;
// without it (FP32 phase of the mixed form) the loop stops after such a step.
// State of a solve paused between two iterations (FP64 form, two passes):
// with r, it is everything the next iteration depends on (f and J are
// recomputed at r), so a resumed solve takes exactly the steps the
// uninterrupted one would have.
struct NewtonState {
    double rho;
    int chord_fail;
    int it;
    bool paused;
    bool flat = false;      // a step below the rounding of the residual was taken (tile kernels)
};

template <int n, typename T, bool FINAL, bool WARP = false>
__device__ T newton(const ElemPtr<T>& el, const BasisTab& tab, const T (&xs)[3], T (&r)[3], T (&J)[9], int max_it,
                    bool& converged, NewtonState* st = nullptr, int budget = 0x7fffffff)
{
    static_assert(!WARP || (FINAL && sizeof(T) == 8), "the warp-cooperative solver is the FP64 one");
    auto fJ = [&](const T (&rr)[3], T (&ff)[3], T (&JJ)[9]) {
        if constexpr (WARP) eval_fJ_warp<n>(el, tab, rr, xs, ff, JJ);
        else eval_fJ<n, T>(el, tab, rr, xs, ff, JJ);
    };
    T f[3];
    fJ(r, f, J);
    T phi = T(0.5) * (f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
    T rho = st ? T(st->rho) : T(1);
    int chord_fail = st ? st->chord_fail : 0;   // after two failed chord checks the trust-region rules alone finish
    const int it0 = st ? st->it : 0;
    if (st) st->paused = false;
    converged = true;
    for (int it = it0; it < max_it; ++it) {
        if (st && it - it0 >= budget) {                   // pause: the caller resumes later
            st->rho = (double)rho;
            st->chord_fail = chord_fail;
            st->it = it;
            st->paused = true;
            converged = false;
            return sqrt(T(2) * phi);
        }
        if (!(phi > T(0))) return T(0);
        T d[3];
        const int nfree = gn_step<T>(J, f, r, d);
        if (nfree == 0) return sqrt(T(2) * phi);          // KKT point at a vertex
        const T dn = fmax(fabs(d[0]), fmax(fabs(d[1]), fabs(d[2])));
        if (!(dn > T(0))) return sqrt(T(2) * phi);
        bool full = true;
        if (dn > rho) {
            const T sc = rho / dn;
            d[0] *= sc; d[1] *= sc; d[2] *= sc;
            full = false;
        }
        T rn[3];
        if (box_step<T>(r, d, rn) < T(1)) full = false;
        T s[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) s[b] = rn[b] - r[b];
        const T sn = fmax(fabs(s[0]), fmax(fabs(s[1]), fabs(s[2])));
        if (!(sn > T(0))) return sqrt(T(2) * phi);
        // a small unconstrained Newton step: quadratic convergence from here
        if (full && nfree == 3 && dn <= Lim<T>::quick && chord_fail < 2) {
            if constexpr (!FINAL) {
                r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                return sqrt(T(2) * phi);
            } else {
                T rc[3] = {rn[0], rn[1], rn[2]};
                T res;
                if (chord64<n, WARP>(el, tab, xs, rc, J, res, 3)) {
                    r[0] = rc[0]; r[1] = rc[1]; r[2] = rc[2];
                    return res;
                }
                r[0] = rc[0]; r[1] = rc[1]; r[2] = rc[2];   // not yet converged: refresh J
                ++chord_fail;
                fJ(r, f, J);
                phi = T(0.5) * (f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
                continue;
            }
        }
        T mf[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) mf[a] = f[a] + J[3 * a] * s[0] + J[3 * a + 1] * s[1] + J[3 * a + 2] * s[2];
        const T pred = phi - T(0.5) * (mf[0] * mf[0] + mf[1] * mf[1] + mf[2] * mf[2]);
        T fn[3], Jn[9];
        fJ(rn, fn, Jn);
        const T phin = T(0.5) * (fn[0] * fn[0] + fn[1] * fn[1] + fn[2] * fn[2]);
        if (sn <= Lim<T>::stop) {
            if (phin <= phi) {
                r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
#pragma unroll
                for (int q = 0; q < 9; ++q) J[q] = Jn[q];
                phi = phin;
            }
            return sqrt(T(2) * phi);
        }
        if (phin < phi) {
            const T ratio = pred > T(0) ? (phi - phin) / pred : T(0);
            r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
#pragma unroll
            for (int q = 0; q < 9; ++q) J[q] = Jn[q];
            f[0] = fn[0]; f[1] = fn[1]; f[2] = fn[2];
            phi = phin;
            if (ratio > T(0.75) && sn >= T(0.99) * rho) rho = fmin(T(2) * rho, T(2));
            else if (ratio < T(0.25)) rho = T(0.25) * sn;
        } else {
            rho = T(0.25) * sn;
            // a radius collapsed below the rounding level: converged as far as
            // this precision resolves (the FP32 phase only supplies a start)
            if (rho < Lim<T>::rho_min) return sqrt(T(2) * phi);
        }
    }
    converged = false;                                     // iteration cap
    return sqrt(T(2) * phi);
}

// nearest mapped GLL node (ties: lowest node index) -> its reference coordinates
template <int n, typename T>
__device__ __forceinline__ void seed_nearest(const ElemPtr<T>& el, const BasisTab& tab, const T (&xs)[3], T (&r)[3])
{
    constexpr int n3 = n * n * n;
    T best = T(INFINITY);
    int bq = 0;
    if constexpr (sizeof(T) == 4 && n3 % 4 == 0) {
        // four nodes per 16-byte load (every element's rows start 16-byte aligned)
        const float4* X0 = reinterpret_cast<const float4*>(el.X0);
        const float4* X1 = reinterpret_cast<const float4*>(el.X1);
        const float4* X2 = reinterpret_cast<const float4*>(el.X2);
#pragma unroll 2
        for (int q4 = 0; q4 < n3 / 4; ++q4) {
            const float4 a = __ldg(X0 + q4), b = __ldg(X1 + q4), c = __ldg(X2 + q4);
            const float ax[4] = {a.x, a.y, a.z, a.w}, bx[4] = {b.x, b.y, b.z, b.w}, cx[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const T dx = ax[m] - xs[0], dy = bx[m] - xs[1], dz = cx[m] - xs[2];
                const T d2 = dx * dx + dy * dy + dz * dz;
                if (d2 < best) {
                    best = d2;
                    bq = 4 * q4 + m;
                }
            }
        }
    } else {
#pragma unroll 4
        for (int q = 0; q < n3; ++q) {
            const T dx = __ldg(el.X0 + q) - xs[0];
            const T dy = __ldg(el.X1 + q) - xs[1];
            const T dz = __ldg(el.X2 + q) - xs[2];
            const T d2 = dx * dx + dy * dy + dz * dz;
            if (d2 < best) {
                best = d2;
                bq = q;
            }
        }
    }
    const int i = bq % n, j = (bq / n) % n, k = bq / (n * n);
    r[0] = Tab<T>::xi(tab)[i];
    r[1] = Tab<T>::xi(tab)[j];
    r[2] = Tab<T>::xi(tab)[k];
}

struct NewtonArgs {
    const int32_t* dcount;  // device-side pair total (capped by cap)
    int64_t E;
    const int32_t* order;
    const int32_t* pair_elem;
    const int32_t* pair_pt;
    int64_t P;
    const double* pts;
    const double* coords;
    const float* coords32;
    const float* coords32lo;  // mixed form: low parts of the element-local coordinates
    const ElemBox* boxes;
    double* pres;
    double* prst;
    int64_t cap;
    double reject32;      // mixed: reject after FP32 when residual > reject32 * h_e
    int max_newton;
    int refine;           // mixed: compensated residuals per pair before the FP64 fallback
    int first_pass;       // iterations (tile kernels: evaluations) of the first pass
    unsigned long long* stats;  // optional path counters (profiling): [0] rejected after FP32,
                                // [1] FP32 not converged, [2] FP64 step converged, [3] sent to the fallback
    const int32_t* warm_elem;   // optional [P]: each point's element at the previous mesh position
    const double* warm_rst;     // [3][P]: its reference coordinates there
    int32_t* fb_count;          // mixed form: number of pairs sent to the FP64 fallback (zeroed before)
    int32_t* fb_list;           // their slots, the first fb_cap of them (batch groups: from the group's
    int64_t fb_cap;             //   first sorted position, capacity = the group's pairs)
    // batch groups: the group's pairs are the sorted positions [*s_lo, *s_hi)
    // (null: [0, live pairs)); pair_elem - ebase indexes the group's arrays
    const int32_t* s_lo;
    const int32_t* s_hi;
    int32_t ebase;
    int32_t* queue;             // work-queue counter (zeroed before the launch); null = grid-stride
    int tile;                   // sorted positions per work item (a multiple of 32)
    double2* pstate;            // state of solves paused after the first pass's budget, per pair: rho and
                                //   chord_fail + 4 it (k_newton) or + 4 flat + 8 it (tile kernels); null = one pass
    const unsigned char* digits;   // tile kernels: the elements' node digits (fp_tile.cuh)
    int rows;                   // tile kernels: sorted positions per warp, 1..32; 0: from the count on the device
    int32_t* pause_list;        // tile kernels: result positions of the solves paused after first_pass
    int32_t* pause_count;       //   evaluations (with pstate), capacity = all pairs; their number (zeroed before)
    bool resume;                // FP64 tile kernel: run the paused solves instead
    int list_blocks;            // mixed tile kernels, second launch: its first blocks run the listed solves
    int list_spread;            //   a short list is spread over this many of them
    float* jst;                 // [9][cap] mixed tile kernels in two launches: the FP32 phase's Jacobian
    bool walk;                  // pair results (pres, prst, pstate) at sorted positions s (coalesced);
                                //   otherwise at pair slots q.  Fallback lists hold the same index.
};

// where pair s / q keeps its results, and the pair of a listed index
__device__ __forceinline__ int64_t result_slot(const NewtonArgs& A, int64_t s, int32_t q) { return A.walk ? s : q; }
__device__ __forceinline__ int32_t listed_pair(const NewtonArgs& A, int64_t t) { return A.walk ? A.order[t] : (int32_t)t; }

struct PairRange {
    int64_t s0, s1;
};

__device__ __forceinline__ PairRange pair_range(const NewtonArgs& A)
{
    if (A.s_lo) return {(int64_t)*A.s_lo, (int64_t)*A.s_hi};
    return {0, live_pairs(A.dcount, A.cap)};
}

// Visit the sorted pair positions of the range: grid-stride over a fixed
// grid, or (queue) work items of `tile` consecutive positions that whole
// warps draw from a device counter, so a warp whose pairs converged fast
// takes the next item instead of idling (pairs of one element stay together
// in an item).  The counter only grows; no warp waits on another.
template <typename Fn>
__device__ __forceinline__ void for_each_pair(const NewtonArgs& A, const PairRange& R, Fn&& fn)
{
    if (!A.queue) {
        for (int64_t s = R.s0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < R.s1;
             s += (int64_t)gridDim.x * blockDim.x)
            fn(s);
        return;
    }
    const int lane = threadIdx.x & 31;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(A.queue, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        const int64_t t0 = R.s0 + (int64_t)item * A.tile;
        if (t0 >= R.s1) break;
        const int64_t t1 = t0 + A.tile < R.s1 ? t0 + A.tile : R.s1;
        for (int64_t s = t0 + lane; s < t1; s += 32) fn(s);
    }
}

// the same for whole warps: each takes `rows` consecutive positions at a
// time, as block `bid` of nb (one call site, so that the solver is compiled
// once)
template <typename Fn>
__device__ __forceinline__ void for_each_rows(const NewtonArgs& A, const PairRange& R, int rows, bool queue, int bid, int nb,
                                              Fn&& fn)
{
    int64_t s = R.s0, end = R.s0, stride = rows;
    if (!queue) {
        s += ((bid * (int64_t)blockDim.x + threadIdx.x) >> 5) * rows;
        end = R.s1;
        stride = (((int64_t)nb * blockDim.x) >> 5) * rows;
    }
    for (;; s += stride) {
        if (s >= end) {
            if (!queue) break;
            int item = 0;
            if ((threadIdx.x & 31) == 0) item = atomicAdd(A.queue, 1);
            item = __shfl_sync(0xffffffffu, item, 0);
            s = R.s0 + (int64_t)item * A.tile;
            if (s >= R.s1) break;
            end = s + A.tile < R.s1 ? s + A.tile : R.s1;
        }
        fn(s, s + rows < end ? s + rows : end);
    }
}

// warm start (moving meshes): a pair whose element is the point's previous
// element starts from the previous reference coordinates, clamped to the
// reference cube, instead of the nearest node.  Only the start changes; a
// non-finite previous value falls back to the nearest node.
__device__ __forceinline__ bool warm_seed(const NewtonArgs& A, int64_t p, int e, double (&r)[3])
{
    if (!A.warm_elem || A.warm_elem[p] != e) return false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double v = A.warm_rst[a * A.P + p];
        if (!(fabs(v) <= 2.0)) return false;
        r[a] = fmin(1.0, fmax(-1.0, v));
    }
    return true;
}

// FP32 value of a reference coordinate that is +-1 only when r is exactly +-1
__device__ __forceinline__ float f32_inside(double v)
{
    float f = (float)v;
    if (f >= 1.0f && v < 1.0) f = 0.99999994f;       // largest float below 1
    if (f <= -1.0f && v > -1.0) f = -0.99999994f;
    return f;
}

// ---- compensated FP32 residual for the refinement steps of the mixed form ----
// x_local(r) - x*_local with node offsets X - c held as float pairs (hi, lo),
// basis values computed in FP64 and split, products formed exactly in their
// leading part and summed with error-free two-sums (about 48 significant
// bits in element-local units).  Runs on the FP32 pipes.
// Lagrange basis at r in double-float arithmetic, on the FP32 pipes: r split
// into (hi, lo), each factor r - xi_m by an error-free difference, the
// prefix / suffix products and the normalisers c_i as double-float products.
// About 2^-45 absolute error on the basis values (measured against
// extended-precision products: 2.7e-14 at worst, 2e-15 rms, for N = 7),
// against 2^-48 for an FP64 basis split afterwards; the residuals that use it
// only steer and confirm the final Newton steps.
template <int n>
__device__ __forceinline__ void lagrange_h_df(const df& r, const BasisTab& tab, float (&hh)[n], float (&hl)[n])
{
    df dm[n];
#pragma unroll
    for (int m = 0; m < n; ++m) dm[m] = df_sub(r, df{tab.xif[m], tab.xil[m]});
    df pre[n];
    pre[0] = {1.0f, 0.0f};
#pragma unroll
    for (int i = 1; i < n; ++i) pre[i] = df_mul(pre[i - 1], dm[i - 1]);
    df suf = {1.0f, 0.0f};
#pragma unroll
    for (int i = n - 1; i >= 0; --i) {
        const df t = df_mul(df{tab.cif[i], tab.cil[i]}, df_mul(pre[i], suf));
        hh[i] = t.hi;
        hl[i] = t.lo;
        suf = df_mul(suf, dm[i]);
    }
}

template <int n>
__device__ __forceinline__ void resid_df(const ElemPtr<float>& hi, const ElemPtr<float>& lo, const BasisTab& tab,
                                         const double (&r)[3], const double (&xl)[3], float (&f)[3])
{
    float rh[n], rl[n], sh[n], sl[n], th[n], tl[n];
    lagrange_h_df<n>(df_split(r[0]), tab, rh, rl);
    lagrange_h_df<n>(df_split(r[1]), tab, sh, sl);
    lagrange_h_df<n>(df_split(r[2]), tab, th, tl);
    df acc[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        df ck[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const int off = n * (j + n * k);
            df u[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {             // three coordinates: three independent chains
                const float* Xh = (a == 0 ? hi.X0 : (a == 1 ? hi.X1 : hi.X2)) + off;
                const float* Xl = (a == 0 ? lo.X0 : (a == 1 ? lo.X1 : lo.X2)) + off;
                float vh[n], vl[n];
                load_row<n>(Xh, vh);
                load_row<n>(Xl, vl);
                u[a] = row_df<n>(vh, vl, rh, rl);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) df_fma_acc(ck[a], u[a].hi, u[a].lo, sh[j], sl[j]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            df_norm(ck[a]);
            df_fma_acc(acc[a], ck[a].hi, ck[a].lo, th[k], tl[k]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float xh = (float)xl[a];
        const float xlo = (float)(xl[a] - (double)xh);
        f[a] = (acc[a].hi - xh) + (acc[a].lo - xlo);
    }
}

// Threshold of the final step's convergence check on a double-float
// residual: 1e-13 in r, raised to the rounding level of a step where that is
// larger.  The residual is accurate to a few units of 2^-48 of the
// element-local coordinates (|x - c_e| <= h_e), which a step J^-1 f turns
// into ||J^-1|| times as much in r; 2^-46 h_e ||J^-1||_inf bounds that noise.
__device__ __forceinline__ double chord_tol_df(const double (&J)[9], double he)
{
    const double C00 = J[4] * J[8] - J[5] * J[7], C01 = J[5] * J[6] - J[3] * J[8], C02 = J[3] * J[7] - J[4] * J[6];
    const double det = J[0] * C00 + J[1] * C01 + J[2] * C02;
    if (!(fabs(det) > 0.0) || !isfinite(det)) return Lim<double>::chord;
    const double C10 = J[2] * J[7] - J[1] * J[8], C11 = J[0] * J[8] - J[2] * J[6], C12 = J[1] * J[6] - J[0] * J[7];
    const double C20 = J[1] * J[5] - J[2] * J[4], C21 = J[2] * J[3] - J[0] * J[5], C22 = J[0] * J[4] - J[1] * J[3];
    const double rows = fmax(fabs(C00) + fabs(C10) + fabs(C20),
                             fmax(fabs(C01) + fabs(C11) + fabs(C21), fabs(C02) + fabs(C12) + fabs(C22)));
    return fmax(Lim<double>::chord, 1.4210854715202004e-14 * he * rows / fabs(det));
}

// final steps of the mixed form: at most NewtonArgs::refine double-float
// residuals (3 by default); a step of at most kConfirm (computed in FP32) is
// re-solved in FP64; an FP64 step of at most kTake chord tolerances is taken
// without another residual (see solve_mixed)
constexpr double kConfirm = 1e-10;
constexpr double kTake = 1e3;

}  // namespace fpg
