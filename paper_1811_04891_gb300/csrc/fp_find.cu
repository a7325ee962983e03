// fp_find.cu -- point location (Sec. 2.1, findpts) as a pair stream.
//
//  1. k_screen<false>  per point: hash cell -> candidate list, session
//                      filter (sub != tag), axis box, box in the element's
//                      affine frame; count the survivors.
//  2. scan             per-point pair offsets.
//  3. k_screen<true>   write the (point, element) pairs in point order.
//  4. k_ehist / scan / k_escatter   counting sort of the pairs by element, so
//                      neighbouring threads work on the same element and its
//                      geometry is served by broadcast loads from L1.
//  5. Newton         per pair: seed at the nearest mapped GLL node (or the
//                      point's previous (e, r) on a moving mesh), then
//                      box-constrained trust-region Newton on
//                      ||x^e(r) - x*||^2 (fp_solve.cu).  Most orders run
//                      k_newton_tile<n,KIND>, on the tensor cores, from an
//                      affine start; the others k_newton<n> (FP64 form) or
//                      k_newton_mixed<n>: the early iterations in FP32 on
//                      element-local coordinates, a compensated refinement
//                      and one FP64 step.  k_newton64_full<n> finishes the
//                      pairs of the mixed form that were not confirmed.
//  6. k_rank<n,3>      per point: classify its pairs (INSIDE / BORDER), lowest
//                      element id within a subdomain, owner = argmax of the
//                      interpolated distance field D^k with lower-id tie band.
#include <algorithm>

#include "fp_common.cuh"
#include "fp_internal.h"
#include "fp_newton.cuh"

namespace fpg {

// ---------------------------------------------------------------------------
// screening
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool inside_boxes(const ElemBox* __restrict__ bp, double x, double y, double z)
{
    const double* b = reinterpret_cast<const double*>(bp);
    // ElemBox layout: c[0..2], Ai[3..11], olo[12..14], ohi[15..17], blo[18..20], bhi[21..23]
    if (x < __ldg(b + 18) || x > __ldg(b + 21) || y < __ldg(b + 19) || y > __ldg(b + 22) ||
        z < __ldg(b + 20) || z > __ldg(b + 23))
        return false;
    const double dx = x - __ldg(b + 0), dy = y - __ldg(b + 1), dz = z - __ldg(b + 2);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double v = __ldg(b + 3 + 3 * a) * dx + __ldg(b + 4 + 3 * a) * dy + __ldg(b + 5 + 3 * a) * dz;
        if (v < __ldg(b + 12 + a) || v > __ldg(b + 15 + a)) return false;
    }
    return true;
}

__device__ __forceinline__ bool inside_boxes32(const ElemBox32* __restrict__ bp, float x, float y, float z)
{
    const float* b = reinterpret_cast<const float*>(bp);
    // ElemBox32 layout: c[0..2], Ai[3..11], olo[12..14], ohi[15..17], blo[18..20], bhi[21..23]
    if (x < __ldg(b + 18) || x > __ldg(b + 21) || y < __ldg(b + 19) || y > __ldg(b + 22) ||
        z < __ldg(b + 20) || z > __ldg(b + 23))
        return false;
    const float dx = x - __ldg(b + 0), dy = y - __ldg(b + 1), dz = z - __ldg(b + 2);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float v = __ldg(b + 3 + 3 * a) * dx + __ldg(b + 4 + 3 * a) * dy + __ldg(b + 5 + 3 * a) * dz;
        if (v < __ldg(b + 12 + a) || v > __ldg(b + 15 + a)) return false;
    }
    return true;
}

struct ScreenArgs {
    int64_t P;
    const double* pts;
    const int32_t* qsess;
    const int32_t* sub;
    const ElemBox* boxes;
    const ElemBox32* boxes32;
    HashGrid g;
    const int32_t* cell_start;
    const int32_t* cell_elems;
    int32_t* cnt;
    const int32_t* off;
    int32_t* pair_elem;
    int32_t* pair_pt;
    int64_t cap;          // pair capacity: pairs at positions >= cap are not written
    int64_t stride;       // row stride of pts (and offset of y, z rows); 0 means P
    int32_t pt_base;      // added to the point index written into pair_pt
    int32_t elem_base;    // added to the element index written into pair_elem
    uint32_t* mask;       // optional [P]: the count pass records which entries of the point's cell list
                          //   passed (bit q - start), so the emit pass need not test them again;
                          //   kMaskOverflow marks lists longer than 31 entries (tested again)
};

constexpr uint32_t kMaskOverflow = 0x80000000u;

// the hash cell of a point (-1: not finite or outside the grid); the FP32
// screen hashes in FP32
template <bool F32>
__device__ __forceinline__ int64_t hash_cell(const HashGrid& g, double x, double y, double z)
{
    if (!(isfinite(x) && isfinite(y) && isfinite(z))) return -1;
    double u0, u1, u2;
    if (F32) {
        u0 = (double)(((float)x - (float)g.org[0]) * (float)g.inv[0]);
        u1 = (double)(((float)y - (float)g.org[1]) * (float)g.inv[1]);
        u2 = (double)(((float)z - (float)g.org[2]) * (float)g.inv[2]);
    } else {
        u0 = (x - g.org[0]) * g.inv[0];
        u1 = (y - g.org[1]) * g.inv[1];
        u2 = (z - g.org[2]) * g.inv[2];
    }
    if (!(u0 >= 0.0 && u1 >= 0.0 && u2 >= 0.0 && u0 <= (double)g.dim[0] && u1 <= (double)g.dim[1] &&
          u2 <= (double)g.dim[2]))
        return -1;
    const int i = min((int)u0, g.dim[0] - 1);
    const int j = min((int)u1, g.dim[1] - 1);
    const int k = min((int)u2, g.dim[2] - 1);
    return i + (int64_t)g.dim[0] * (j + (int64_t)g.dim[1] * k);
}

template <bool EMIT, bool F32>
__device__ __forceinline__ void screen_point(const ScreenArgs& A, int64_t p)
{
    const int64_t ld = A.stride ? A.stride : A.P;
    const double x = A.pts[p], y = A.pts[ld + p], z = A.pts[2 * ld + p];
    const int tag = A.qsess ? A.qsess[p] : -1;
    int c = 0;
    int base = EMIT ? A.off[p] : 0;
    uint32_t m = 0;
    if (EMIT && A.mask) m = A.mask[p];
    if (EMIT && A.mask && !(m & kMaskOverflow)) {
        // the count pass found these entries of the point's cell list
        if (m) {
            const int b = __ldg(A.cell_start + hash_cell<F32>(A.g, x, y, z));
            while (m) {
                const int bit = __ffs(m) - 1;
                m &= m - 1;
                if (base + c < A.cap) {
                    A.pair_elem[base + c] = A.elem_base + __ldg(A.cell_elems + b + bit);
                    A.pair_pt[base + c] = A.pt_base + (int32_t)p;
                }
                ++c;
            }
        }
        return;
    }
    const int64_t cell = hash_cell<F32>(A.g, x, y, z);
    if (cell >= 0) {
        const int b = __ldg(A.cell_start + cell), en = __ldg(A.cell_start + cell + 1);
        if (!EMIT && en - b > 31) m = kMaskOverflow;
        for (int q = b; q < en; ++q) {
            const int e = __ldg(A.cell_elems + q);
            if (tag >= 0 && __ldg(A.sub + e) == tag) continue;
            if (F32) {
                if (!inside_boxes32(A.boxes32 + e, (float)x, (float)y, (float)z)) continue;
            } else if (!inside_boxes(A.boxes + e, x, y, z)) {
                continue;
            }
            if (EMIT && base + c < A.cap) {
                A.pair_elem[base + c] = A.elem_base + e;
                A.pair_pt[base + c] = A.pt_base + (int32_t)p;
            }
            if (!EMIT && !(m & kMaskOverflow)) m |= 1u << (q - b);
            ++c;
        }
    }
    if (!EMIT) {
        A.cnt[p] = c;
        if (A.mask) A.mask[p] = m;
    }
}

template <bool EMIT, bool F32>
__global__ void __launch_bounds__(256) k_screen(ScreenArgs A)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= A.P) return;
    screen_point<EMIT, F32>(A, p);
}

// Batches: one thread per point of all instances; the point's instance (the
// last one whose first point is <= p) gives the hash grid, boxes and element
// numbering it is screened against.
template <bool EMIT, bool F32>
__global__ void __launch_bounds__(256) k_bscreen(BScreenArgs B)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= B.P) return;
    int lo = 0, hi = B.ninst;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(B.p0 + mid) <= p) lo = mid;
        else hi = mid;
    }
    const BInst& I = B.inst[lo];
    ScreenArgs A;
    A.P = B.P;
    A.pts = B.pts;
    A.qsess = nullptr;
    A.sub = I.sub;
    A.boxes = I.boxes;
    A.boxes32 = I.boxes32;
    A.g = I.g;
    A.cell_start = I.cell_start;
    A.cell_elems = I.cell_elems;
    A.cnt = B.cnt;
    A.off = B.off;
    A.pair_elem = B.pair_elem;
    A.pair_pt = B.pair_pt;
    A.cap = B.cap;
    A.stride = B.P;
    A.pt_base = 0;
    A.elem_base = I.ebase;
    A.mask = B.mask;
    screen_point<EMIT, F32>(A, p);
}

cudaError_t launch_bscreen(const BScreenArgs& b, bool emit, bool f32, cudaStream_t s)
{
    if (b.P == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((b.P + 255) / 256);
    if (emit) {
        if (f32) k_bscreen<true, true><<<grid, 256, 0, s>>>(b);
        else k_bscreen<true, false><<<grid, 256, 0, s>>>(b);
    } else {
        if (f32) k_bscreen<false, true><<<grid, 256, 0, s>>>(b);
        else k_bscreen<false, false><<<grid, 256, 0, s>>>(b);
    }
    count_launch();
    return cudaGetLastError();
}

__global__ void k_ehist(const int32_t* __restrict__ dcount, int64_t cap, const int32_t* __restrict__ pair_elem,
                        int32_t* __restrict__ ecount)
{
    const int64_t npairs = live_pairs(dcount, cap);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < npairs; q += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(ecount + pair_elem[q], 1);
}

__global__ void k_escatter(const int32_t* __restrict__ dcount, int64_t cap, const int32_t* __restrict__ pair_elem,
                           const int32_t* __restrict__ estart, int32_t* __restrict__ cursor, int32_t* __restrict__ order,
                           int32_t* __restrict__ inv)
{
    const int64_t npairs = live_pairs(dcount, cap);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < npairs; q += (int64_t)gridDim.x * blockDim.x) {
        const int e = pair_elem[q];
        const int pos = estart[e] + atomicAdd(cursor + e, 1);
        order[pos] = (int32_t)q;
        if (inv) inv[q] = pos;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static ScreenArgs screen_args(const FindArgs& a)
{
    ScreenArgs s;
    s.P = a.P;
    s.pts = a.pts;
    s.qsess = a.qsess;
    s.sub = a.sub;
    s.boxes = a.boxes;
    s.boxes32 = a.boxes32;
    s.g = *a.grid;
    s.cell_start = a.cell_start;
    s.cell_elems = a.cell_elems;
    s.cnt = a.cnt;
    s.off = a.off;
    s.pair_elem = a.pair_elem;
    s.pair_pt = a.pair_pt;
    s.cap = a.cap;
    s.stride = a.pts_stride;
    s.pt_base = a.pt_base;
    s.elem_base = a.elem_base;
    s.mask = a.smask;
    return s;
}

cudaError_t find_count(const FindArgs& a, const BasisTab&, const FindParams&, cudaStream_t s)
{
    ScreenArgs sa = screen_args(a);
    if (a.boxes32)
        k_screen<false, true><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    else
        k_screen<false, false><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    count_launch();
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    return scan_exclusive(a.cnt, a.off, a.P, a.scan_tmp, s);
}

cudaError_t find_screen_count(const FindArgs& a, cudaStream_t s)
{
    ScreenArgs sa = screen_args(a);
    if (a.boxes32)
        k_screen<false, true><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    else
        k_screen<false, false><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    count_launch();
    return cudaGetLastError();
}

cudaError_t find_emit(const FindArgs& a, cudaStream_t s)
{
    ScreenArgs sa = screen_args(a);
    if (a.boxes32)
        k_screen<true, true><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    else
        k_screen<true, false><<<(unsigned)((a.P + 255) / 256), 256, 0, s>>>(sa);
    count_launch();
    return cudaGetLastError();
}

// grid for `work` items; with a persistent block count the kernels loop
// grid-stride over a count that only the device knows
static unsigned grid_for(int64_t work, int block, int persistent)
{
    int64_t g = (work + block - 1) / block;
    if (persistent > 0 && g > persistent) g = persistent;
    return (unsigned)(g < 1 ? 1 : g);
}

cudaError_t find_sort(const FindArgs& a, int64_t npairs, cudaStream_t s)
{
    cudaError_t err = cudaSuccess;
    if (npairs > 0) {
        if (a.ev[0]) cudaEventRecord(a.ev[0], s);
        err = cudaMemsetAsync(a.ecount, 0, sizeof(int32_t) * a.E, s);
        if (err != cudaSuccess) return err;
        const unsigned g256 = grid_for(npairs, 256, a.persistent_blocks ? 4 * a.persistent_blocks : 0);
        k_ehist<<<g256, 256, 0, s>>>(a.off + a.P, a.cap, a.pair_elem, a.ecount);
        count_launch();
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        if ((err = scan_exclusive(a.ecount, a.estart, a.E, a.scan_tmp, s)) != cudaSuccess) return err;
        if ((err = cudaMemsetAsync(a.ecount, 0, sizeof(int32_t) * a.E, s)) != cudaSuccess) return err;
        k_escatter<<<g256, 256, 0, s>>>(a.off + a.P, a.cap, a.pair_elem, a.estart, a.ecount, a.order, a.inv);
        count_launch();
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        if (a.ev[1]) cudaEventRecord(a.ev[1], s);
    }
    return err;
}

// ---------------------------------------------------------------------------
// dispatch by order (fp_solve.cu, one object per order)
// ---------------------------------------------------------------------------
#define FP_ORDERS                                                                                                   \
    FP_CASE(2) FP_CASE(3) FP_CASE(4) FP_CASE(5) FP_CASE(6) FP_CASE(7) FP_CASE(8) FP_CASE(9) FP_CASE(10) FP_CASE(11) \
    FP_CASE(12) FP_CASE(13) FP_CASE(14) FP_CASE(15) FP_CASE(16)

#define FP_CASE(NN)                                                                                                     \
    cudaError_t solve_order_##NN(const FindArgs&, int64_t, const BasisTab&, const FindParams&, int, cudaStream_t);      \
    cudaError_t newton_order_##NN(const FindArgs&, int64_t, const BasisTab&, const FindParams&, int, unsigned,          \
                                  cudaStream_t);                                                                        \
    int newton_fit_order_##NN(bool, int);                                                                               \
    cudaError_t digits_order_##NN(bool, int64_t, const double*, ElemBox*, unsigned char*, const BasisTab&, cudaStream_t); \
    int64_t digits_bytes_order_##NN(bool);
FP_ORDERS
#undef FP_CASE

// Newton + classification (+ fused evaluation) on pairs already in `a.order` (no pair sort).
cudaError_t find_solve_unsorted(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp,
                                int block, cudaStream_t s)
{
    switch (a.n) {
#define FP_CASE(NN) case NN: return solve_order_##NN(a, npairs, tab, fp, block, s);
        FP_ORDERS
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t find_solve(const FindArgs& a, int64_t npairs, const BasisTab& tab, const FindParams& fp, int block,
                       cudaStream_t s)
{
    const cudaError_t err = find_sort(a, npairs, s);
    return err != cudaSuccess ? err : find_solve_unsorted(a, npairs, tab, fp, block, s);
}

// Newton stage of one order-n group of a batch (a.s_lo / a.s_hi / a.ebase
// set), on `grid` blocks of `block` threads drawing work items of a.tile
// sorted positions from the counter a.queue.
cudaError_t find_newton_group(const FindArgs& a, const BasisTab& tab, const FindParams& fp, int block, unsigned grid,
                              cudaStream_t s)
{
    switch (a.n) {
#define FP_CASE(NN) case NN: return newton_order_##NN(a, a.cap, tab, fp, block, grid, s);
        FP_ORDERS
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
}

int newton_blocks_per_sm(int n, bool mixed, int block)
{
    switch (n) {
#define FP_CASE(NN) case NN: return newton_fit_order_##NN(mixed, block);
        FP_ORDERS
#undef FP_CASE
        default: return 1;
    }
}

cudaError_t launch_digits(int n, bool mixed, int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig,
                          const BasisTab& tab, cudaStream_t s)
{
    switch (n) {
#define FP_CASE(NN) case NN: return digits_order_##NN(mixed, E, coords, boxes, dig, tab, s);
        FP_ORDERS
#undef FP_CASE
        default: return cudaErrorInvalidValue;
    }
}

int64_t tile_digits_bytes(int n, bool mixed)
{
    switch (n) {
#define FP_CASE(NN) case NN: return digits_bytes_order_##NN(mixed);
        FP_ORDERS
#undef FP_CASE
        default: return 0;
    }
}

}  // namespace fpg
