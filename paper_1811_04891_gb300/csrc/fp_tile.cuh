// fp_tile.cuh -- the element map of Sec. 2.1's Newton solve on the tensor
// cores: one warp evaluates x^e(r) and its Jacobian at up to 32 pairs.
//
// What bounds it and why this split.  One thread per pair evaluates the map by
// sum factorisation: n^3 multiply-adds per coordinate for the first
// contraction, which is all of its time (FP64 form: the FP64 pipe, 2
// multiply-adds per clock and SM; mixed form: 12 FP32 operations for each
// double-float term).  That contraction is a matrix product when the pairs of
// one element are taken together:
//     c[pair][a,k] = sum_{i,j} (h_i(r) h_j(s))[pair][ij] * x_a[ij][k]
// with n^2 products per pair on the left and the element's nodes on the
// right, and only 3 n values per pair are left to contract with h_k(t).
//
// Exactness.  Both factors are cut into signed 10-bit digits (fixed point:
// the basis products lie in [-1,1], the node offsets x - c_e are scaled by a
// power of two per element and coordinate into [-1/2,1/2], so that a thin
// direction of a stretched element keeps all its bits), which FP16 holds exactly.  A
// product of two digits has at most 19 bits, and the FP32 accumulators add
// products of equal weight exactly as long as a sum stays below 2^24.  Orders
// 0 and 1 do (one factor's first digits add up to at most 512 times the
// Lebesgue constant squared, 100 products of 2^17 the other way); for the
// others, sums of n^2 products of digits of either sign, it is a matter of
// odds: 2^23 is the largest seen over 200 random points for N = 3 to 9, 2^24
// is more than 10 standard deviations.  What is left is the last digit's
// rounding and the orders left out.  FP64 form: 6 digits and orders 0..5,
// 2^-58 of the element's size, below an FP64 sum's own rounding (error of x(r)
// against extended precision, relative to half the element's width, N = 7,
// width 0.1: 2e-16 rms; by FP64 sum factorisation 3e-16 for coordinates
// around zero, 3e-15 around 0.5; with 5 digits 3e-15).  Mixed form: 5 digits
// and orders 0..5 for its compensated residuals (1.6e-14 rms, of which 1.5e-14
// from the double-float basis; 1.7e-14 on float pairs of the coordinates,
// 2.0e-14 without order 5), 3 digits and orders 0..2, about 2^-27, for its
// FP32 phase.  A row's sums do not depend on the other
// rows, so a pair's result does not depend on which pairs share its warp, on
// the block size, or on the entry point.
//
// Layout.  A warp takes `rows` consecutive element-sorted pairs, at most 32;
// lane l keeps pair l's Newton state and evaluates its Lagrange bases.  The
// pairs are two 16-row tiles: the lanes build the left factor's digits in
// mma.m16n8k16 fragments and loop over the elements among the pairs (rows of
// other elements masked to zero).  The nodes' digits are laid out once per
// mesh in fragment order, so a fragment is one coalesced load; with three
// digits the next one is fetched while the current one is multiplied.  The
// FP64 form takes dx/dr and dx/ds from the same node digits with h_i' h_j and
// h_i h_j' on the left: a third of the memory, set-up time and L2 traffic of
// digits of the derivatives for two more left factors.  Tiles of 128 pairs
// per tcgen05.mma would leave most rows empty (1 to 300 pairs per element are
// typical), and the 16-row form is not bound by the tensor pipe (18 % busy in
// the FP64 form's first pass, 30 % in the mixed form's two launches): the FP64
// form is by the FP64 pipe (78 %: bases, columns, last contraction, 3x3
// solves; 16 clocks of an SM a warp's operation), the mixed form by issue and
// one warp's chain (46 % and 39 % of the issue slots with 13 and 14 of 16
// warps).
//
// Measured (fp_find, N = 7, before = one thread per pair): 1.0e7 points in
// 32,768 elements, mixed form, this stage 25.8 -> 16.7 ms; 3.0e5 points in
// 1,000 elements, FP64 form, whole find 21.7 -> 2.6 ms; 1,501 points in 216
// elements, N = 6, FP64 form, 1.95 -> 0.43 ms.
#pragma once
#include <cuda_fp16.h>

#include <type_traits>

#include "fp_common.cuh"
#include "fp_internal.h"
#include "fp_newton.cuh"

namespace fpg {

constexpr int kTileRows = 32;          // pairs of a warp, at most
constexpr unsigned kFull = 0xffffffffu;

template <int n>
struct TileDim {
    static_assert(is_tile_order(n, false) || is_tile_order(n, true), "other orders keep one thread per pair");
    static constexpr int n2 = n * n;
    static constexpr int KC = (n2 + 15) / 16;            // k16 steps over (i,j)
    static constexpr int NT = (3 * n + 7) / 8;           // 8-column tiles over (a,k)
    static constexpr int JP = (16 * KC + n - 1) / n;     // j values including the zero padding
};

// Shared memory of one warp: the basis values h_i(r), h_j(s), h_k(t), h_k'(t)
// (FP64 form: also h_i'(r) and h_j'(s)) of its 32 rows, the left factor's digits of one 16-row tile (fragment
// order), the columns c of one tile, and the results (x, dx/dr, dx/ds in three
// coordinates; dx/dt takes the place of a row's h_k'(t)).  Row strides of 34 and 18 eight-byte values (36 and
// 20 floats) put the fragment accesses of a half-warp into distinct banks.
template <typename T> struct TileStride {
    static constexpr int H = sizeof(T) == 4 ? 36 : 34, C = sizeof(T) == 4 ? 20 : 18;
};

template <int n, typename T, int S, int NH, int NO>      // NH: 3, 4 or 6 basis arrays, NO: result quantities
struct TileSm {
    using D = TileDim<n>;
    static constexpr int H = TileStride<T>::H;
    static constexpr int HR = 0, HS = HR + n * H, DR = HS + D::JP * H, DS = DR + n * H,
                         HT = NH == 6 ? DS + D::JP * H : DR, DT = HT + n * H, C = NH == 3 ? DT : DT + n * H,
                         OUT = C + 3 * n * TileStride<T>::C, VALS = OUT + 3 * NO * kTileRows;   // (dx/dt: in DT)
    // the digits start on a 16-byte boundary
    static constexpr int DIG = (int)((VALS * sizeof(T) + 15) / 16 * 16);
    static constexpr int BYTES = DIG + (S > 0 ? D::KC * S * 512 : 0);
};

template <int n> using Sm32 = TileSm<n, float, 3, 4, 3>;    // FP32 phase
template <int n> using SmDf = TileSm<n, float2, 0, 3, 1>;   // compensated residual: digits stay in registers
template <int n> using Sm64 = TileSm<n, double, 0, 6, 3>;   // FP64 form: the same

__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t h2bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }

// ---- digits of two neighbouring products (k, k+1) of one row, as FP16 pairs ----
// v = d_0 2^-9 + d_1 2^-19 + ..., each digit rounded to nearest (adding and
// subtracting 1.5 * 2^23 rounds to an integer), every remainder exact
constexpr float kRnd = 12582912.0f;

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

template <int e>
__device__ __forceinline__ constexpr float pow2()
{
    float v = 1.0f;
    for (int i = 0; i < (e < 0 ? -e : e); ++i) v *= e < 0 ? 0.5f : 2.0f;
    return v;
}

template <int e>
__device__ __forceinline__ float2 digit(float2& v)      // the digit of weight 2^-e; v: remainder
{
    const float2 d = __fadd2_rn(__ffma2_rn(v, f2(pow2<e>()), f2(kRnd)), f2(-kRnd));
    v = __ffma2_rn(d, f2(-pow2<-e>()), v);
    return d;
}

__device__ __forceinline__ uint32_t pack_h2(float2 d) { return h2bits(__floats2half2_rn(d.x, d.y)); }

// FP32 products (the mixed form's FP32 phase): 3 digits
__device__ __forceinline__ void digits2(float a0, float b0, float a1, float b1, uint32_t (&o)[3])
{
    float2 v = __fmul2_rn(make_float2(a0, a1), make_float2(b0, b1));
    o[0] = pack_h2(digit<9>(v));
    o[1] = pack_h2(digit<19>(v));
    o[2] = pack_h2(digit<29>(v));
}

// double-float products: exact leading product p, its error and the cross
// terms e; e joins the remainder once p's upper 20 bits are cut off (twice,
// around the third digit, so that no sum of the two loses bits)
__device__ __forceinline__ void digits2(float2 a0, float2 b0, float2 a1, float2 b1, uint32_t (&o)[5])
{
    const float2 ah = make_float2(a0.x, a1.x), al = make_float2(a0.y, a1.y);
    const float2 bh = make_float2(b0.x, b1.x), bl = make_float2(b0.y, b1.y);
    float2 v = __fmul2_rn(ah, bh);
    const float2 e = __ffma2_rn(ah, bl, __ffma2_rn(al, bh, __ffma2_rn(ah, bh, f2_neg(v))));
    o[0] = pack_h2(digit<9>(v));
    o[1] = pack_h2(digit<19>(v));
    const float2 s = __fadd2_rn(v, e);
    const float2 d2 = __fadd2_rn(__ffma2_rn(s, f2(pow2<29>()), f2(kRnd)), f2(-kRnd));
    o[2] = pack_h2(d2);
    v = __fadd2_rn(__ffma2_rn(d2, f2(-pow2<-29>()), v), e);
    o[3] = pack_h2(digit<39>(v));
    o[4] = pack_h2(digit<49>(v));
}

// FP64 form: a basis value in [-1,1] as x 2^-30 + y 2^-60, |y| <= 2^29: the low
// words of the sums with 1.5 2^22 and 1.5 2^-8 (last bits 2^-30 and 2^-60; the
// difference between them is exact)
__device__ __forceinline__ int2 fix60(double h)
{
    const double p = h + 0x1.8p22, q = h + ((0x1.8p22 + 0x1.8p-8) - p);
    return make_int2(__double2loint(p), __double2loint(q));
}

// makes digit s of a fixed-point value of unit 2^-60 the bits 51 - 10 s and up,
// plus 512, rounded to 2^-59
constexpr int64_t kBias60 = 512ll * ((1ll << 51) + (1ll << 41) + (1ll << 31) + (1ll << 21) + (1ll << 11) + (1ll << 1)) + 1;

// the product of two basis values in units of 2^-60 (y y' left out) plus the
// bias, by integer multiply-adds: the FP64 pipe, with 3 operations a product,
// was what bounded the kernel (2.0e6 points, N = 7, whole find and evaluation:
// 26.1 ms)
__device__ __forceinline__ uint64_t product60(int2 a, int2 b)
{
    const int64_t low = (int64_t)a.x * b.y + ((int64_t)a.y * b.x + (1 << 29));
    return (uint64_t)(((int64_t)a.x * b.x + kBias60) + (low >> 30));
}

// v 2^-e in units of 2^-60 (|v| < 2^(e-1)) plus the bias
__device__ __forceinline__ uint64_t fixed60(double v, int e)
{
    const int64_t b = __double_as_longlong(v);
    const int x = (int)((b >> 52) & 0x7ff), sh = 1015 + e - max(x, 1);      // right shift
    const int64_t m = (b & 0xfffffffffffffll) | (x ? 1ll << 52 : 0);
    const int64_t k = sh <= 0 ? m << -sh : sh > 54 ? 0 : (m + (1ll << (sh - 1))) >> sh;
    return (uint64_t)((b < 0 ? -k : k) + kBias60);
}

// three digits of two values, as FP16 pairs: f is the FP16 number 1024 + f
// (bits 0x6400 + f) minus 1536; the first digit of all reaches 512 (11 bits)
template <bool FIRST>
__device__ __forceinline__ void fields3(uint32_t u, uint32_t w, uint32_t* o)
{
    const __half2 off = __floats2half2_rn(1536.0f, 1536.0f);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t v = __byte_perm(u >> (10 * (2 - s)), w >> (10 * (2 - s)), 0x5410);
        v = FIRST && s == 0 ? (v & 0x07ff07ffu) + 0x64006400u : (v & 0x03ff03ffu) | 0x64006400u;
        o[s] = h2bits(__hsub2(*reinterpret_cast<__half2*>(&v), off));
    }
}

// the 6 digits of two biased fixed-point values
__device__ __forceinline__ void fields6(uint64_t u, uint64_t w, uint32_t (&o)[6])
{
    fields3<true>((uint32_t)(u >> 31), (uint32_t)(w >> 31), o);
    fields3<false>((uint32_t)(u >> 1), (uint32_t)(w >> 1), o + 3);
}

__device__ __forceinline__ void digits2(int2 a0, int2 b0, int2 a1, int2 b1, uint32_t (&o)[6])
{
    fields6(product60(a0, b0), product60(a1, b1), o);
}

// ---- the element's nodes as digits, in B-fragment order ----
// per element: the nodes x (KC x NT fragments; 6 digits in the FP64 form, 5 in
// the mixed form) and, mixed form, the nodal values of dx/dr and dx/ds in 3
// digits (the derivative of the interpolant is the interpolant of its nodal
// values), so that x, dx/dr and dx/ds share the left factor h_i h_j.  A
// fragment: 32 lanes x (digits 0,1), 32 lanes x (digits 2,3), ..., an odd last
// digit by itself.  A lane's digit is two registers of two FP16 values.
template <int S> struct FragBytes { static constexpr int v = 32 * 8 * S; };

template <int n, bool MIXED>
struct TileBytes {
    static constexpr int SX = MIXED ? 5 : 6;             // digits of the nodes
    static constexpr int64_t frags = (int64_t)TileDim<n>::KC * TileDim<n>::NT;
    static constexpr int64_t jac = frags * FragBytes<SX>::v, one = MIXED ? frags * FragBytes<3>::v : 0, v = jac + 2 * one;
};

// which rows of a 16-row tile start a new element
__device__ __forceinline__ uint32_t tile_heads(uint32_t heads, int mt) { return ((heads >> (16 * mt)) | 1u) & 0xffffu; }

// digits of rows g and g + 8 of tile mt at k16 step kc, in fragment order
template <int n, int S, typename T>
__device__ __forceinline__ void tile_left(const T* hi, const T* hj, int kc, int mt, uint32_t (&a)[S][4])
{
    constexpr int PS = TileStride<T>::H;
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        const int k0 = 16 * kc + 8 * hf + 2 * q, k1 = k0 + 1;
        const int j0 = k0 / n, j1 = k1 / n, i0 = k0 - n * j0, i1 = k1 - n * j1;
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int row = 16 * mt + g + 8 * rr;
            uint32_t d[S];
            const T b0 = hj[j0 * PS + row], b1 = n % 2 == 0 ? b0 : hj[j1 * PS + row];   // even n: j1 = j0
            digits2(hi[i0 * PS + row], b0, hi[i1 * PS + row], b1, d);
#pragma unroll
            for (int s = 0; s < S; ++s) a[s][2 * hf + rr] = d[s];
        }
    }
}

// a fragment of the right factor: S digits of one 8-column tile, of sb stored
template <int S>
struct RightFrag {
    uint32_t b[S][2];
    __device__ __forceinline__ void load(const unsigned char* __restrict__ F, int sb)
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int u = 0; u + 1 < S; u += 2) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(F + 256 * u) + lane);
            b[u][0] = v.x; b[u][1] = v.y; b[u + 1][0] = v.z; b[u + 1][1] = v.w;
        }
        if constexpr (S % 2 == 1) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(F + 256 * (S - 1)) + (sb > S ? 2 * lane : lane));
            b[S - 1][0] = v.x; b[S - 1][1] = v.y;
        }
    }
    __device__ __forceinline__ void store(unsigned char* F) const
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int u = 0; u + 1 < S; u += 2)
            reinterpret_cast<uint4*>(F + 256 * u)[lane] = make_uint4(b[u][0], b[u][1], b[u + 1][0], b[u + 1][1]);
        if constexpr (S % 2 == 1) reinterpret_cast<uint2*>(F + 256 * (S - 1))[lane] = make_uint2(b[S - 1][0], b[S - 1][1]);
    }
};

// ---- fragments of an element without stored digits ----
// The digits that k_digits lays out, made from the coordinates where they are
// used (with the scales it left in boxes): the same bits for no memory.  m: 0
// the nodes, 1 and 2 (mixed form) the nodal values of dx/dr and dx/ds, whose
// rows of n products are most of the cost.  A find, stored / made here, us:
// N = 7, 4,096 elements, FP64 form 1,000 points 341/439, 400,000 2768/4413;
// mixed form 157/275, 890/7330; N = 9 mixed 1,820/22,966.
struct NodeSource {
    const double* coords;
    const float* coords32;
    const ElemBox* boxes;
    int64_t E;
    const float* der;                  // der[i n + u] = h_u'(xi_i) (mixed form)
};

__device__ __forceinline__ int exp_of(double p) { return ((__double2hiint(p) >> 20) & 0x7ff) - 1023; }
__device__ __forceinline__ int exp_of(float p) { return ((__float_as_int(p) >> 23) & 0xff) - 127; }

// one of the nodal values of dx/dr (st = 1) or dx/ds (st = n): the row through
// v times the derivatives of row `at`
template <int n>
__device__ __forceinline__ float nodal_derivative(const float* der, const float* v, int at, int st)
{
    float w = 0.0f;
#pragma unroll
    for (int u = 0; u < n; ++u) w = fmaf(der[at * n + u], v[u * st], w);
    return w;
}

// rows of the table by the block's first n threads
template <int n>
__device__ __forceinline__ void derivative_table(const BasisTab& tab, float* der)
{
    if (threadIdx.x < n) {
        float h[n], d[n];
        lagrange_hd<n, float>(tab.xif, tab.cif, tab.xif[threadIdx.x], h, d);
#pragma unroll
        for (int m = 0; m < n; ++m) der[threadIdx.x * n + m] = d[m];
    }
}

template <int n, int S>
__device__ __forceinline__ void make_frag(const NodeSource& N, int el, int kc, int t, int m, RightFrag<S>& R)
{
    constexpr int n2 = n * n, n3 = n2 * n;
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int col = 8 * t + g, a = col < n ? 0 : col < 2 * n ? 1 : 2, k = col - a * n;
    const ElemBox& bx = N.boxes[el];
    const int64_t plane = ((int64_t)a * N.E + el) * n3 + n2 * k;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        const int kap = 16 * kc + 8 * hf + 2 * q;
        if (m == 0) {
            uint64_t w[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const bool in = kap + u < n2 && col < 3 * n;
                w[u] = fixed60(in ? __ldg(N.coords + plane + kap + u) - bx.c[a] : 0.0, exp_of(bx.scale) + exp_of(bx.cscale[a]));
            }
            uint32_t d[6];
            fields6(w[0], w[1], d);
#pragma unroll
            for (int s = 0; s < S; ++s) R.b[s][hf] = d[s];
        } else if constexpr (S == 3) {
            float v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int x = kap + u, at = m == 1 ? x % n : x / n, st = m == 1 ? 1 : n;
                const bool in = x < n2 && col < 3 * n;
                v[u] = in ? ldexpf(nodal_derivative<n>(N.der, N.coords32 + plane + x - at * st, at, st),
                                   -(exp_of(bx.scale) + exp_of(bx.jscale[m - 1][a])))
                          : 0.0f;
            }
            uint32_t d[3];
            digits2(v[0], 1.0f, v[1], 1.0f, d);
#pragma unroll
            for (int s = 0; s < S; ++s) R.b[s][hf] = d[s];
        }
    }
}

// acc[o][t] += the order-o products of S left digits and the S right digits of
// tile t; FINE: order S joins the sums of order S - 1, its right digits scaled
// by 2^-10
template <int n, int S, int O, bool FINE>
__device__ __forceinline__ void mma_digits(const uint32_t (&a)[S][4], const RightFrag<S>& R, int t,
                                           float (&acc)[O][TileDim<n>::NT][4])
{
#pragma unroll
    for (int u = 0; u < S; ++u)
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (s + u < O) mma_16816(acc[s + u][t], a[s], R.b[u][0], R.b[u][1]);
    if constexpr (FINE) {
        static_assert(O == S, "the next order is S");
        const __half2 sc = __floats2half2_rn(pow2<-10>(), pow2<-10>());
        auto down = [&](uint32_t d) { return h2bits(__hmul2(*reinterpret_cast<const __half2*>(&d), sc)); };
#pragma unroll
        for (int u = 1; u < S; ++u) mma_16816(acc[S - 1][t], a[S - u], down(R.b[u][0]), down(R.b[u][1]));
    }
}

// acc = the digit products of a 16-row tile over all k16 steps.  left(kc, a)
// gives the tile's digits, right(el, kc, t, R) an element's fragments.  One
// element among the rows: the next step's fragments are fetched while the
// current ones are multiplied (three digits: they fit the registers).
// Several: each element's rows in turn, the others masked to zero.
template <int n, int S, int O, bool FINE, typename Left, typename Right>
__device__ __forceinline__ void tile_gemm(Left&& left, Right&& right, uint32_t heads, uint32_t need, int e, int mt,
                                          float (&acc)[O][TileDim<n>::NT][4])
{
    using D = TileDim<n>;
    const int lane = threadIdx.x & 31, g = lane >> 2;
#pragma unroll
    for (int o = 0; o < O; ++o)
#pragma unroll
        for (int t = 0; t < D::NT; ++t)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[o][t][v] = 0.0f;
    // heads of the elements with a row that wants a value
    uint32_t hs = 0;
    for (uint32_t hm = heads; hm;) {
        const int h = __ffs(hm) - 1;
        hm &= hm - 1;
        const int nx = hm ? __ffs(hm) - 1 : 16;
        if ((need >> h) & ((1u << (nx - h)) - 1u)) hs |= 1u << h;
    }
    if (!hs) return;
    auto elem = [&](int h) { return __shfl_sync(kFull, e, 16 * mt + h); };
    RightFrag<S> next[S == 3 ? D::NT : 1];
    auto fetch = [&](int h, int kc) {
        const int el = elem(h);
#pragma unroll
        for (int t = 0; t < D::NT; ++t) right(el, kc, t, next[t]);
    };
    if constexpr (S == 3) {
        fetch(__ffs(hs) - 1, 0);
        if (heads == 1u) {
#pragma unroll 1
            for (int kc = 0; kc < D::KC; ++kc) {
                RightFrag<S> R[D::NT];
#pragma unroll
                for (int t = 0; t < D::NT; ++t) R[t] = next[t];
                if (kc + 1 < D::KC) fetch(0, kc + 1);
                uint32_t a[S][4];
                left(kc, a);
#pragma unroll
                for (int t = 0; t < D::NT; ++t) mma_digits<n, S, O, FINE>(a, R[t], t, acc);
            }
            return;
        }
    }
#pragma unroll 1
    for (int kc = 0; kc < D::KC; ++kc) {
        uint32_t a[S][4];
        left(kc, a);
        uint32_t hm = hs;
#pragma unroll 1
        while (hm) {
            const int h = __ffs(hm) - 1;
            hm &= hm - 1;
            const uint32_t after = heads & ~((2u << h) - 1u);
            const int nx = after ? __ffs(after) - 1 : 16;
            uint32_t am[S][4];
            const uint32_t m0 = g >= h && g < nx ? ~0u : 0u, m1 = g + 8 >= h && g + 8 < nx ? ~0u : 0u;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                am[s][0] = a[s][0] & m0;
                am[s][1] = a[s][1] & m1;
                am[s][2] = a[s][2] & m0;
                am[s][3] = a[s][3] & m1;
            }
            if constexpr (S == 3) {
                RightFrag<S> R[D::NT];
#pragma unroll
                for (int t = 0; t < D::NT; ++t) R[t] = next[t];
                if (hm || kc + 1 < D::KC) fetch(__ffs(hm ? hm : hs) - 1, hm ? kc : kc + 1);
#pragma unroll
                for (int t = 0; t < D::NT; ++t) mma_digits<n, S, O, FINE>(am, R[t], t, acc);
            } else {
                const int el = elem(h);
#pragma unroll
                for (int t = 0; t < D::NT; ++t) {
                    RightFrag<S> R;
                    right(el, kc, t, R);
                    mma_digits<n, S, O, FINE>(am, R, t, acc);
                }
            }
        }
    }
}

// ---- a column's value from its order sums ----
// FP32 phase: one float in units of the element's scale
__device__ __forceinline__ float column(float a0, float a1, float a2)
{
    return fmaf(a2, pow2<-38>(), fmaf(a1, pow2<-28>(), a0 * pow2<-18>()));
}

// double-float, two columns at once: the sums of orders 0 and 1 and then
// order 2 by error-free two-sums
__device__ __forceinline__ df2 column_df(float2 a0, float2 a1, float2 a2, float2 a3, float2 a4)
{
    const float2 t = __ffma2_rn(a1, f2(pow2<-10>()), a0);
    const float2 e1 = __ffma2_rn(a1, f2(pow2<-10>()), f2_neg(__fadd2_rn(t, f2_neg(a0))));
    const float2 c = __fmul2_rn(a2, f2(pow2<-20>()));
    const float2 s = __fadd2_rn(t, c);
    const float2 bb = __fadd2_rn(s, f2_neg(t));
    const float2 e2 = __fadd2_rn(__fadd2_rn(t, f2_neg(__fadd2_rn(s, f2_neg(bb)))), __fadd2_rn(c, f2_neg(bb)));
    const float2 lo = __ffma2_rn(a4, f2(pow2<-40>()), __ffma2_rn(a3, f2(pow2<-30>()), __fadd2_rn(e1, e2)));
    return {__fmul2_rn(s, f2(pow2<-18>())), __fmul2_rn(lo, f2(pow2<-18>()))};
}

// FP64, in units of 2^-58: the sums are whole numbers; orders 0 and 1 make one
// in units of 2^-28, the others (order 5 rounded) one in units of 2^-58, and
// their bits in 1.5 2^82 and 1.5 2^52 give the two as FP64 numbers, added with
// one rounding
__device__ __forceinline__ double column_f64(float a0, float a1, float a2, float a3, float a4, float a5)
{
    const int64_t hi = (int64_t)__float2int_rn(a0) * 1024 + __float2int_rn(a1);
    const int64_t lo = ((int64_t)__float2int_rn(a2) * 1024 + __float2int_rn(a3)) * 1024 + __float2int_rn(a4) +
                       __float2int_rn(a5 * pow2<-10>());
    const double H = __longlong_as_double(hi + 0x4518000000000000ll), W = __longlong_as_double(lo + 0x4338000000000000ll);
    return (H - (0x1.8p82 + 0x1.8p52)) + W;
}

// ---- collective evaluations: lane l holds row l ----
template <int n, bool FLY>
struct TileCtx {
    unsigned char* sm;                 // this warp's shared memory
    const unsigned char* dig;          // stored digits
    NodeSource src;                    // FLY: what they are made from
    uint32_t heads;                    // rows whose element differs from the row before
    int e;                             // the row's element
    const ElemBox* bx;

    // fragment (kc, t) of quantity m (see make_frag): S digits of those stored
    template <int S, bool MIXED>
    __device__ __forceinline__ void frag(int el, int kc, int t, int m, RightFrag<S>& R) const
    {
        using TB = TileBytes<n, MIXED>;
        if constexpr (FLY) {
            make_frag<n, S>(src, el, kc, t, m, R);
        } else {
            const int sb = MIXED && m > 0 ? 3 : TB::SX;
            R.load(dig + (int64_t)el * TB::v + (MIXED && m > 0 ? TB::jac + (m - 1) * TB::one : 0) +
                       (kc * TileDim<n>::NT + t) * (FragBytes<1>::v * sb), sb);
        }
    }
};

// store one direction's values of this lane's row; the j padding is zero
template <int n, typename T>
__device__ __forceinline__ void store_dir(T* p, bool pad, const T (&h)[n])
{
#pragma unroll
    for (int i = 0; i < n; ++i) p[i * TileStride<T>::H] = h[i];
    if (pad)
#pragma unroll
        for (int i = n; i < TileDim<n>::JP; ++i) p[i * TileStride<T>::H] = T{};
}

// sum_k w_k c[a n + k] of a 16-row tile into the results: a = 0
// (lanes < 16) and 1 (lanes >= 16) in one pass, then a = 2; with `both` also
// the sums with the second weights, over these
template <int n, typename T>
__device__ __forceinline__ void contract_out(T* out, bool both, const T* c, const T* w, T* w2)
{
    constexpr int PS = TileStride<T>::C, HS = TileStride<T>::H;
    const int lane = threadIdx.x & 31, row = lane & 15, a01 = lane >> 4;
    T s = T(0), s2 = T(0), t = T(0), t2 = T(0);
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const T wk = w[k * HS + row], ck = c[(a01 * n + k) * PS + row], ck2 = c[(2 * n + k) * PS + row];
        s = fma(wk, ck, s);
        s2 = fma(wk, ck2, s2);
        if (both) {
            const T vk = w2[k * HS + row];
            t = fma(vk, ck, t);
            t2 = fma(vk, ck2, t2);
        }
    }
    out[a01 * kTileRows + row] = s;
    if (lane < 16) out[2 * kTileRows + row] = s2;
    if (both) {
        __syncwarp();                                     // both of a row's lanes have read w2
        w2[a01 * HS + row] = t;
        if (lane < 16) w2[2 * HS + row] = t2;
    }
}

// exact FP32 -> FP64 by integer operations: the FP64 pipe takes 16 clocks of
// an SM for a warp's conversion, these take two
__device__ __forceinline__ double widen(float f)
{
    const uint32_t b = (uint32_t)__float_as_int(f), m = b & 0x7fffffffu;
    const uint32_t hi = m < 0x00800000u ? 0u : ((m >> 3) + 0x38000000u);
    return __hiloint2double((int)(hi | (b & 0x80000000u)), m < 0x00800000u ? 0 : (int)(b << 29));
}

// a power of two f times 2^e (FP64: e goes into the exponent)
template <typename T, int e = 0>
__device__ __forceinline__ T scale_of(float f)
{
    if constexpr (sizeof(T) == 8) return __hiloint2double((__float_as_int(f) >> 3) + 0x38000000 + e * 0x100000, 0);
    else return f * pow2<e>();
}

// |h_i'| <= N^2 <= 2^kDerivExp on the reference interval (Markov's inequality
// for |h_i| <= 1): the derivatives' factor in the FP64 form
template <int n> constexpr int kDerivExp = n <= 4 ? 4 : n <= 5 ? 4 : n <= 6 ? 5 : n <= 9 ? 6 : 7;

// map x(r) in the element's frame and scale, and its Jacobian: T = float (to
// FP32 accuracy, the mixed form's FP32 phase) or double (FP64 form)
template <int n, typename T, bool FLY>
__device__ __forceinline__ void tile_fJ(const TileCtx<n, FLY>& X, const BasisTab& tab, uint32_t need, bool jac,
                                        const T (&r)[3], T (&x)[3], T (&J)[9])
{
    constexpr bool F64 = sizeof(T) == 8;
    using D = TileDim<n>;
    using L = std::conditional_t<F64, Sm64<n>, Sm32<n>>;
    constexpr int S = F64 ? 6 : 3, O = S, CS = TileStride<T>::C;
    static_assert((n - 1) * (n - 1) <= 1 << kDerivExp<n>, "derivatives are scaled into [-1,1]");
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    T* sm = reinterpret_cast<T*>(X.sm);
    uint4* dg = reinterpret_cast<uint4*>(X.sm + L::DIG);
    if constexpr (F64) {
        // h_i(r), h_j(s) and their derivatives in fixed point, h_k(t) and h_k'(t) in FP64
        int2* fx = reinterpret_cast<int2*>(sm);
#pragma unroll 1
        for (int d = 0; d < 3; ++d) {
            const T rd = d == 0 ? r[0] : d == 1 ? r[1] : r[2];
            T h[n], dh[n];
            if (jac) lagrange_hd<n, T>(tab.xi, tab.ci, rd, h, dh);
            else lagrange_h<n, T>(tab.xi, tab.ci, rd, h);
            if (d == 2) {
                store_dir<n, T>(sm + L::HT + lane, false, h);
                if (jac) store_dir<n, T>(sm + L::DT + lane, false, dh);
            } else {
                int2 v[n];
#pragma unroll
                for (int i = 0; i < n; ++i) v[i] = fix60(h[i]);
                store_dir<n, int2>(fx + (d == 0 ? L::HR : L::HS) + lane, d == 1, v);
                if (jac) {
#pragma unroll
                    for (int i = 0; i < n; ++i) v[i] = fix60(dh[i] * T(pow2<-kDerivExp<n>>()));
                    store_dir<n, int2>(fx + (d == 0 ? L::DR : L::DS) + lane, d == 1, v);
                }
            }
        }
    } else {
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {
            T h[n];
            lagrange_h<n, T>(tab.xif, tab.cif, d == 0 ? r[0] : r[1], h);
            store_dir<n, T>(sm + (d == 0 ? L::HR : L::HS) + lane, d == 1, h);
        }
        T h[n], dh[n];
        lagrange_hd<n, T>(tab.xif, tab.cif, r[2], h, dh);
        store_dir<n, T>(sm + L::DT + lane, false, dh);
        store_dir<n, T>(sm + L::HT + lane, false, h);
    }
    __syncwarp();
#pragma unroll 1
    for (int mt = 0; mt < 2; ++mt) {
        const uint32_t nd = (need >> (16 * mt)) & 0xffffu, hd = tile_heads(X.heads, mt);
        if (!nd) continue;
        if constexpr (!F64) {
#pragma unroll 1
            for (int kc = 0; kc < D::KC; ++kc) {
                uint32_t a[S][4];
                tile_left<n, S, T>(sm + L::HR, sm + L::HS, kc, mt, a);
#pragma unroll
                for (int s = 0; s < S; ++s) dg[(kc * S + s) * 32 + lane] = make_uint4(a[s][0], a[s][1], a[s][2], a[s][3]);
            }
        }
        // each lane reads back the digits it wrote itself: no barrier
#pragma unroll 1
        for (int m = 0; m < (jac ? 3 : 1); ++m) {         // x, dx/dr, dx/ds
            float acc[O][D::NT][4];
            auto left = [&](int kc, uint32_t (&a)[S][4]) {
                if constexpr (F64) {
                    const int2* fx = reinterpret_cast<const int2*>(sm);
                    tile_left<n, S, int2>(fx + (m == 1 ? L::DR : L::HR), fx + (m == 2 ? L::DS : L::HS), kc, mt, a);
                } else {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        const uint4 v = dg[(kc * S + s) * 32 + lane];
                        a[s][0] = v.x; a[s][1] = v.y; a[s][2] = v.z; a[s][3] = v.w;
                    }
                }
            };
            tile_gemm<n, S, O, false>(
                left, [&](int el, int kc, int t, RightFrag<S>& R) { X.template frag<S, !F64>(el, kc, t, F64 ? 0 : m, R); }, hd,
                nd, X.e, mt, acc);
            T* C = sm + L::C;
#pragma unroll
            for (int t = 0; t < D::NT; ++t)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int col = 8 * t + 2 * q + (v & 1), row = g + 8 * (v >> 1);
                    if (col < 3 * n) {
                        if constexpr (F64)
                            C[col * CS + row] = column_f64(acc[0][t][v], acc[1][t][v], acc[2][t][v], acc[3][t][v],
                                                           acc[4][t][v], acc[5][t][v]);
                        else
                            C[col * CS + row] = column(acc[0][t][v], acc[1][t][v], acc[2][t][v]);
                    }
                }
            __syncwarp();
            T* out = sm + L::OUT + 16 * mt;
            contract_out<n, T>(out + 3 * m * kTileRows, jac && m == 0, C, sm + L::HT + 16 * mt, sm + L::DT + 16 * mt);
            __syncwarp();
        }
    }
    // from each coordinate's own scale (FP64: and the columns' unit) to the element's
    constexpr int unit = F64 ? -58 : 0;
    const T* out = sm + L::OUT + lane;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const T cs = scale_of<T, unit>(X.bx->cscale[a]);
        x[a] = out[a * kTileRows] * cs;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            T js = cs;
            if (b < 2) {
                if constexpr (F64) js = scale_of<T, unit + kDerivExp<n>>(X.bx->cscale[a]);
                else js = X.bx->jscale[b][a];
            }
            J[3 * a + b] = (b < 2 ? out[(3 + 3 * b + a) * kTileRows] : sm[L::DT + a * TileStride<T>::H + lane]) * js;
        }
    }
    __syncwarp();
}

// residual x(r) - x* as double-float, rounded to FP32 (r and xl, the point in
// the element's frame and scale, as float pairs)
template <int n, bool FLY>
__device__ __forceinline__ void tile_f_df(const TileCtx<n, FLY>& X, const BasisTab& tab, uint32_t need, const df (&r)[3],
                                          const df (&xl)[3], float (&f)[3])
{
    using D = TileDim<n>;
    using L = SmDf<n>;
    constexpr int CS = TileStride<float2>::C, HP = TileStride<float2>::H;
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    float2* sm = reinterpret_cast<float2*>(X.sm);
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        float hh[n], hl[n];
        lagrange_h_df<n>(df{d == 0 ? r[0].hi : d == 1 ? r[1].hi : r[2].hi, d == 0 ? r[0].lo : d == 1 ? r[1].lo : r[2].lo}, tab,
                         hh, hl);
        float2 h[n];
#pragma unroll
        for (int i = 0; i < n; ++i) h[i] = make_float2(hh[i], hl[i]);
        store_dir<n, float2>(sm + (d == 0 ? L::HR : d == 1 ? L::HS : L::HT) + lane, d == 1, h);
    }
    __syncwarp();
#pragma unroll 1
    for (int mt = 0; mt < 2; ++mt) {
        const uint32_t nd = (need >> (16 * mt)) & 0xffffu, hd = tile_heads(X.heads, mt);
        if (!nd) continue;
        float acc[5][D::NT][4];
        tile_gemm<n, 5, 5, true>(
            [&](int kc, uint32_t (&a)[5][4]) { tile_left<n, 5, float2>(sm + L::HR, sm + L::HS, kc, mt, a); },
            [&](int el, int kc, int t, RightFrag<5>& R) { X.template frag<5, true>(el, kc, t, 0, R); }, hd, nd, X.e, mt, acc);
        float2* C = sm + L::C;
#pragma unroll
        for (int t = 0; t < D::NT; ++t)
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                auto at = [&](int o) { return make_float2(acc[o][t][2 * rr], acc[o][t][2 * rr + 1]); };
                const df2 c = column_df(at(0), at(1), at(2), at(3), at(4));
                const int col = 8 * t + 2 * q, row = g + 8 * rr;
                if (col < 3 * n) C[col * CS + row] = make_float2(c.hi.x, c.lo.x);
                if (col + 1 < 3 * n) C[(col + 1) * CS + row] = make_float2(c.hi.y, c.lo.y);
            }
        __syncwarp();
        const int row = lane & 15, a01 = lane >> 4;
        const float2* w = sm + L::HT + 16 * mt + row;
        df u = {0.0f, 0.0f}, u2 = {0.0f, 0.0f};
#pragma unroll 2
        for (int k = 0; k < n; ++k) {
            const float2 h = w[k * HP], c = C[(a01 * n + k) * CS + row], c2 = C[(2 * n + k) * CS + row];
            df_fma_acc(u, c.x, c.y, h.x, h.y);
            df_fma_acc(u2, c2.x, c2.y, h.x, h.y);
        }
        float2* out = sm + L::OUT + 16 * mt + row;
        out[a01 * kTileRows] = make_float2(u.hi, u.lo);
        if (lane < 16) out[2 * kTileRows] = make_float2(u2.hi, u2.lo);
        __syncwarp();
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float2 y = sm[L::OUT + a * kTileRows + lane];
        const float cs = X.bx->cscale[a];
        f[a] = (y.x * cs - xl[a].hi) + (y.y * cs - xl[a].lo);
    }
    __syncwarp();
}

// nearest mapped GLL node of each flagged row (ties: lowest node index), the
// warp scanning one row's element at a time; used where an element's map is
// far from its affine frame
template <int n, typename T>
__device__ __forceinline__ void tile_seed_nearest(const T* __restrict__ coords, int64_t E, uint32_t rows, int e,
                                                  const T (&xs)[3], const T* __restrict__ xi, T (&r)[3])
{
    constexpr int n3 = n * n * n;
    const int lane = threadIdx.x & 31;
    while (rows) {
        const int row = __ffs(rows) - 1;
        rows &= rows - 1;
        const int64_t el = __shfl_sync(kFull, e, row);
        const T x = __shfl_sync(kFull, xs[0], row), y = __shfl_sync(kFull, xs[1], row), z = __shfl_sync(kFull, xs[2], row);
        const T *X0 = coords + el * n3, *X1 = coords + (E + el) * n3, *X2 = coords + (2 * E + el) * n3;
        T best = T(INFINITY);
        int bq = 0;
#pragma unroll 1
        for (int q = lane; q < n3; q += 32) {
            const T dx = __ldg(X0 + q) - x, dy = __ldg(X1 + q) - y, dz = __ldg(X2 + q) - z;
            const T d2 = dx * dx + dy * dy + dz * dz;
            if (d2 < best) {
                best = d2;
                bq = q;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T ob = __shfl_xor_sync(kFull, best, o);
            const int oq = __shfl_xor_sync(kFull, bq, o);
            if (ob < best || (ob == best && oq < bq)) {
                best = ob;
                bq = oq;
            }
        }
        if (lane == row) {
            r[0] = xi[bq % n];
            r[1] = xi[(bq / n) % n];
            r[2] = xi[bq / (n * n)];
        }
    }
}

// An element whose nodes lie within this distance (in reference units) of its
// vertex-averaged affine frame starts its solves at the affine inverse
// y = A^-1 (x* - c), clamped to the cube: closer than the nearest node
// (spacing 0.13 to 0.42 at n = 8) at the cost of nine multiply-adds instead
// of a scan of n^3 nodes, and one Newton iteration less.  A coordinate that
// could lie on a bound (within the deviation, or 1/64) starts on it, as the
// nearest node would: a start a rounding error off the bound would have every
// step cut short there.
constexpr float kAffineSeed = 0.25f;

__device__ __forceinline__ void affine_seed(const ElemBox& bx, const double (&xc)[3], double (&r)[3])
{
    const float v[3] = {(float)xc[0], (float)xc[1], (float)xc[2]};
    const float near = 1.0f - fmaxf(0.015625f, (float)bx.dev);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float y = (float)bx.Ai[3 * a] * v[0] + (float)bx.Ai[3 * a + 1] * v[1] + (float)bx.Ai[3 * a + 2] * v[2];
        r[a] = y > near ? 1.0 : y < -near ? -1.0 : (double)y;
    }
}

// Coordinates on a bound, as bits (b: lower, 3 + b: upper).  A coordinate
// within the rounding level of a step counts as on the bound: kept off it,
// its next outward step would cut the whole step short at a length set by
// rounding, and the solve could stop there.
template <typename T> constexpr T kOnBound = T(1) - (sizeof(T) == 8 ? T(3e-14) : T(5e-7));

template <typename T>
__device__ __forceinline__ int on_bounds(const T (&r)[3])
{
    int on = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) on |= (r[b] <= -kOnBound<T> ? 1 << b : 0) | (r[b] >= kOnBound<T> ? 8 << b : 0);
    return on;
}

// gn_step (fp_newton.cuh) with one 3x3 solve for every case: J d = -f with
// all coordinates free, else the normal equations with the active rows those
// of the identity.  (The instruction cache of an SM holds less than these
// kernels' code if every case has its own.)  on: on_bounds.  Returns the
// number of free coordinates.
template <typename T>
__device__ __forceinline__ int gn_tile(const T (&J)[9], const T (&f)[3], int on, T (&d)[3])
{
    T g[3] = {T(0), T(0), T(0)};
    int act = 0, nfree = 3;
    if (on) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            g[b] = J[b] * f[0] + J[3 + b] * f[1] + J[6 + b] * f[2];
            if (((on >> b) & 1 && g[b] > T(0)) || ((on >> (3 + b)) & 1 && g[b] < T(0))) act |= 1 << b;
        }
    }
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
        nfree = 3 - __popc(act);
        d[0] = d[1] = d[2] = T(0);
        if (nfree == 0) break;
        T M[9], v[3];
        if (act == 0) {
#pragma unroll
            for (int k = 0; k < 9; ++k) M[k] = J[k];
            v[0] = f[0]; v[1] = f[1]; v[2] = f[2];
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                v[a] = act & (1 << a) ? T(0) : g[a];
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    M[3 * a + b] = act & ((1 << a) | (1 << b)) ? (a == b ? T(1) : T(0))
                                                               : J[a] * J[b] + J[3 + a] * J[3 + b] + J[6 + a] * J[6 + b];
            }
        }
        const T C00 = M[4] * M[8] - M[5] * M[7], C01 = M[5] * M[6] - M[3] * M[8], C02 = M[3] * M[7] - M[4] * M[6];
        const T det = M[0] * C00 + M[1] * C01 + M[2] * C02;
        if (act == 0 ? det != T(0) && isfinite(det) : det > T(0)) {
            const T id = T(-1) / det;
            d[0] = (C00 * v[0] + (M[2] * M[7] - M[1] * M[8]) * v[1] + (M[1] * M[5] - M[2] * M[4]) * v[2]) * id;
            d[1] = (C01 * v[0] + (M[0] * M[8] - M[2] * M[6]) * v[1] + (M[2] * M[3] - M[0] * M[5]) * v[2]) * id;
            d[2] = (C02 * v[0] + (M[1] * M[6] - M[0] * M[7]) * v[1] + (M[0] * M[4] - M[1] * M[3]) * v[2]) * id;
        } else {                                          // singular: steepest descent
#pragma unroll
            for (int b = 0; b < 3; ++b)
                d[b] = act & (1 << b) ? T(0) : -(J[b] * f[0] + J[3 + b] * f[1] + J[6 + b] * f[2]);
        }
        const int was = act;
#pragma unroll
        for (int b = 0; b < 3; ++b)
            if (((on >> b) & 1 && d[b] < T(0)) || ((on >> (3 + b)) & 1 && d[b] > T(0))) act |= 1 << b;
        if (act == was) break;
    }
    return nfree;
}

// box_step with one division a coordinate, and none where the step stays
// inside: the new point lands exactly on the bound it was cut at
template <typename T>
__device__ __forceinline__ T box_tile(const T (&r)[3], const T (&d)[3], T (&rn)[3])
{
    bool cut = false;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        rn[b] = r[b] + d[b];
        cut = cut || !(fabs(rn[b]) <= T(1));
    }
    if (!cut) return T(1);
    T t = T(1), tb[3];
#pragma unroll 1
    for (int b = 0; b < 3; ++b) {
        const T rb = b == 0 ? r[0] : b == 1 ? r[1] : r[2], db = b == 0 ? d[0] : b == 1 ? d[1] : d[2];
        const T v = fabs(rb + db) > T(1) ? ((db > T(0) ? T(1) : T(-1)) - rb) / db : T(2);
        if (b == 0) tb[0] = v;
        else if (b == 1) tb[1] = v;
        else tb[2] = v;
        t = fmin(t, v);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        T v = r[b] + t * d[b];
        if (t < T(1) && tb[b] == t) v = d[b] > T(0) ? T(1) : T(-1);
        rn[b] = fmin(T(1), fmax(T(-1), v));
    }
    return t;
}

// ||J^-1||_inf in FP32: it only scales thresholds
template <typename T>
__device__ __forceinline__ float inv_norm(const T (&Jd)[9])
{
    float J[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) J[k] = (float)Jd[k];
    const float C00 = J[4] * J[8] - J[5] * J[7], C01 = J[5] * J[6] - J[3] * J[8], C02 = J[3] * J[7] - J[4] * J[6];
    const float det = J[0] * C00 + J[1] * C01 + J[2] * C02;
    const float C10 = J[2] * J[7] - J[1] * J[8], C11 = J[0] * J[8] - J[2] * J[6], C12 = J[1] * J[6] - J[0] * J[7];
    const float C20 = J[1] * J[5] - J[2] * J[4], C21 = J[2] * J[3] - J[0] * J[5], C22 = J[0] * J[4] - J[1] * J[3];
    const float rows = fmaxf(fabsf(C00) + fabsf(C10) + fabsf(C20),
                             fmaxf(fabsf(C01) + fabsf(C11) + fabsf(C21), fabsf(C02) + fabsf(C12) + fabsf(C22)));
    const float v = rows / fabsf(det);
    return isfinite(v) ? v : 0.0f;
}

// ---- FP64 form: the steps of newton<n, double, true> as a state machine, so
// that the rows of a warp share their evaluations ----
template <int n, bool FLY>
__device__ __forceinline__ void tile_solve_f64(const TileCtx<n, FLY>& X, const NewtonArgs& A, const BasisTab& tab, bool active,
                                               const double (&xl)[3], double xmax,
                                               double (&r)[3], double& res2, NewtonState& st)
{
    enum { FIRST, TRIAL, CHORD, REFRESH, DONE };
    int state = active ? FIRST : DONE;
    double rn[3] = {r[0], r[1], r[2]};                    // where the next evaluation is wanted
    double f[3] = {0, 0, 0}, J[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    double phi = 0.0, rho = st.rho, pred = 0.0, sn = 0.0, ctol = 0.0;
    int chord_fail = st.chord_fail, it = st.it, chord_it = 0;
    bool flat = st.flat;
    st.paused = false;
#pragma unroll 1
    for (int trip = 1;; ++trip) {
        const uint32_t wj = __ballot_sync(kFull, state == FIRST || state == TRIAL || state == REFRESH);
        const uint32_t wf = __ballot_sync(kFull, state == CHORD);
        if (!(wj | wf)) break;
        double fn[3], Jn[9];
        tile_fJ<n, double>(X, tab, wj | wf, wj != 0, rn, fn, Jn);
        if (state == DONE) continue;
#pragma unroll
        for (int a = 0; a < 3; ++a) fn[a] -= xl[a];
        const double f2n = fn[0] * fn[0] + fn[1] * fn[1] + fn[2] * fn[2];
        const bool chord = state == CHORD;
        bool end = false;
        if (chord) {                                      // value-only residual with the fixed Jacobian (chord64)
            res2 = f2n;
            end = !(f2n > 0.0);
        } else {
            const double phin = 0.5 * f2n;
            bool take = true;
            if (state == TRIAL) {
                const double dec = phi - phin;
                if (sn <= Lim<double>::stop) {
                    take = dec >= 0.0;
                    end = true;
                } else {
                    // a change below the rounding of phi (|f| times 2^-48)
                    // says nothing about the step: it is taken, and the
                    // second of them ends the solve
                    const bool level = dec * dec <= 2.5e-29 * phi;
                    take = dec > 0.0 || level;
                    end = level && flat;
                    flat = flat || level;
                    if (take) {
                        // actual over predicted decrease above 3/4, below 1/4
                        if (pred > 0.0 && dec > 0.75 * pred && sn >= 0.99 * rho) rho = fmin(2.0 * rho, 2.0);
                        else if (dec > 0.0 && dec < 0.25 * pred) rho = 0.25 * sn;
                    } else {
                        rho = 0.25 * sn;
                        end = rho < Lim<double>::rho_min;
                    }
                }
            }
            if (state != FIRST) ++it;
            if (take) {
                r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                f[0] = fn[0]; f[1] = fn[1]; f[2] = fn[2];
#pragma unroll
                for (int k = 0; k < 9; ++k) J[k] = Jn[k];
                phi = phin;
            }
            res2 = 2.0 * phi;
            end = end || it >= A.max_newton || !(phi > 0.0);
        }
        if (!end) {
            // the next step: from r with its own J, or from the chord's point
            const double at[3] = {chord ? rn[0] : r[0], chord ? rn[1] : r[1], chord ? rn[2] : r[2]};
            const double fa[3] = {chord ? fn[0] : f[0], chord ? fn[1] : f[1], chord ? fn[2] : f[2]};
            double d[3];
            const int nfree = gn_tile<double>(J, fa, on_bounds(at), d);
            const double dn = fmax(fabs(d[0]), fmax(fabs(d[1]), fabs(d[2])));
            end = nfree == 0 || (!chord && !(dn > 0.0));
            if (!end) {
                bool full = true;
                if (!chord && dn > rho) {
                    const double sc = rho / dn;
                    d[0] *= sc; d[1] *= sc; d[2] *= sc;
                    full = false;
                }
                double to[3];
                if (box_tile<double>(at, d, to) < 1.0) full = false;
                const double s[3] = {to[0] - at[0], to[1] - at[1], to[2] - at[2]};
                sn = fmax(fabs(s[0]), fmax(fabs(s[1]), fabs(s[2])));
                if (chord) {
                    end = sn <= ctol;
                    if (!end && ++chord_it >= 3) {        // not yet converged: refresh J
                        ++chord_fail;
                        state = REFRESH;
                    }
                } else {
                    end = !(sn > 0.0);
                    if (full && nfree == 3 && dn <= Lim<double>::quick && chord_fail < 2) {
                        // 2 eps |x*| ||J^-1||_inf: see chord_tol3
                        ctol = fmax(Lim<double>::chord, 4.440892098500626e-16 * xmax * (double)inv_norm<double>(J));
                        chord_it = 0;
                        state = CHORD;
                    } else {
                        double m2 = 0.0;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const double mf = f[a] + J[3 * a] * s[0] + J[3 * a + 1] * s[1] + J[3 * a + 2] * s[2];
                            m2 += mf * mf;
                        }
                        pred = phi - 0.5 * m2;
                        state = TRIAL;
                    }
                }
                if (!end) {
                    rn[0] = to[0]; rn[1] = to[1]; rn[2] = to[2];
                }
            }
        }
        if (end) {
            if (chord) {
                r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
            }
            state = DONE;
        } else if (trip >= A.first_pass && (state == TRIAL || state == REFRESH)) {
            // a resumed solve evaluates at r first and goes on from there
            if (state == REFRESH) {
                r[0] = rn[0]; r[1] = rn[1]; r[2] = rn[2];
                ++it;
            }
            st = NewtonState{rho, chord_fail, it, true, flat};
            state = DONE;
        }
    }
}

// ---- mixed form: the FP32 phase (newton<n, float, false>) as a state machine ----
// fate: 0 rejected after it, 1 not converged, 3 left to the full FP64 Newton
// (refine = 0; res2 < 0 in the last two).  Returns whether the row goes on to
// the final steps, with r and J from here.
template <int n, bool FLY>
__device__ __forceinline__ bool tile_phase32(const TileCtx<n, FLY>& X, const NewtonArgs& A, const BasisTab& tab, bool active,
                                             const double (&xl)[3], double hes, double (&r)[3],
                                             float (&J)[9], double& res2, int& fate, NewtonState& st)
{
    enum { FIRST, TRIAL, DONE };
    int state = active ? FIRST : DONE;
    float q[3] = {(float)r[0], (float)r[1], (float)r[2]}, qn[3] = {q[0], q[1], q[2]};
    float f[3] = {0, 0, 0};
    float phi = 0.0f, rho = (float)st.rho, pred = 0.0f, sn = 0.0f;
    int it = st.it;
    bool flat = st.flat;
    bool final = false;
    fate = 3;
    st.paused = false;
    res2 = -1.0;
#pragma unroll 1
    for (int trip = 1;; ++trip) {
        const uint32_t want = __ballot_sync(kFull, state != DONE);
        if (!want) break;
        float fn[3], Jn[9];
        tile_fJ<n, float>(X, tab, want, true, qn, fn, Jn);
        if (state == DONE) continue;
#pragma unroll
        for (int a = 0; a < 3; ++a) fn[a] -= (float)xl[a];
        const float phin = 0.5f * (fn[0] * fn[0] + fn[1] * fn[1] + fn[2] * fn[2]);
        bool take = true, end = false, conv = true;
        if (state == TRIAL) {
            const float dec = phi - phin;
            if (sn <= Lim<float>::stop) {
                take = dec >= 0.0f;
                end = true;
            } else {
                // a change below the rounding of phi: see tile_solve_f64
                const bool level = dec * dec <= 1e-13f * phi;
                take = dec > 0.0f || level;
                end = level && flat;
                flat = flat || level;
                if (take) {
                    if (pred > 0.0f && dec > 0.75f * pred && sn >= 0.99f * rho) rho = fminf(2.0f * rho, 2.0f);
                    else if (dec > 0.0f && dec < 0.25f * pred) rho = 0.25f * sn;
                } else {
                    rho = 0.25f * sn;
                    end = rho < Lim<float>::rho_min;
                }
            }
            ++it;
        }
        if (take) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                q[a] = qn[a];
                f[a] = fn[a];
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) J[k] = Jn[k];
            phi = phin;
        }
        if (!end && it >= A.max_newton) {
            end = true;
            conv = false;
        }
        end = end || !(phi > 0.0f);
        if (!end) {
            float d[3];
            const int nfree = gn_tile<float>(J, f, on_bounds(q), d);
            const float dn = fmaxf(fabsf(d[0]), fmaxf(fabsf(d[1]), fabsf(d[2])));
            end = nfree == 0 || !(dn > 0.0f);
            if (!end) {
                bool full = true;
                if (dn > rho) {
                    const float sc = rho / dn;
                    d[0] *= sc; d[1] *= sc; d[2] *= sc;
                    full = false;
                }
                if (box_tile<float>(q, d, qn) < 1.0f) full = false;
                const float s[3] = {qn[0] - q[0], qn[1] - q[1], qn[2] - q[2]};
                sn = fmaxf(fabsf(s[0]), fmaxf(fabsf(s[1]), fabsf(s[2])));
                end = !(sn > 0.0f);
                if (!end && full && nfree == 3 && dn <= Lim<float>::quick) {
                    q[0] = qn[0]; q[1] = qn[1]; q[2] = qn[2];
                    end = true;
                }
                float m2 = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float mf = f[a] + J[3 * a] * s[0] + J[3 * a + 1] * s[1] + J[3 * a + 2] * s[2];
                    m2 += mf * mf;
                }
                pred = phi - 0.5f * m2;
                state = TRIAL;
            }
        }
        if (end) {
            const double r32 = sqrtf(2.0f * phi);
            r[0] = q[0]; r[1] = q[1]; r[2] = q[2];
            if (!conv || !(r32 <= A.reject32 * hes)) {
                res2 = conv ? r32 * r32 : -1.0;
                fate = conv ? 0 : 1;
            } else {
                final = A.refine > 0;
            }
            state = DONE;
        } else if (trip >= A.first_pass) {
            // a resumed solve evaluates at r first and goes on from there
            r[0] = q[0]; r[1] = q[1]; r[2] = q[2];
            st = NewtonState{(double)rho, 0, it, true, flat};
            state = DONE;
        }
    }
    return final;
}

// ---- mixed form: the final steps on compensated residuals (see solve_mixed)
// with the FP32 phase's Jacobian.  fate: 2 finished, 3 left to the full FP64
// Newton (res2 < 0).
// r is carried as a float pair: it starts as an FP32 value, the first step is
// added by an error-free sum, and the sum with the last step is formed in
// FP64.  The FP64 3x3 solve of a small step refines the FP32 solution once
// (residual f + J d in FP64, correction with the FP32 adjugate: relative
// error ~1e-12, far below that of J).  Together ~30 FP64 operations a pair
// instead of ~280, which were 65 % of this phase's time.
// edge: rows that ended the FP32 phase on or near a bound, with active sets
// and cuts; the others have no bound within reach of their steps.  EDGE false
// is the code of the latter alone (it fits the instruction cache). ----
constexpr float kEdge = 0.9999f;

template <int n, bool EDGE, bool FLY>
__device__ __forceinline__ void tile_final(const TileCtx<n, FLY>& X, const NewtonArgs& A, const BasisTab& tab, bool active,
                                           const double (&xl)[3], double hes, double (&r)[3], const float (&J)[9],
                                           double& res2, int& fate)
{
    const bool edge = EDGE && fmax(fabs(r[0]), fmax(fabs(r[1]), fabs(r[2]))) >= (double)kEdge;
    int fin = 0;
    df rp[3], xp[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        rp[a] = df_split(r[a]);
        xp[a] = df_split(xl[a]);
    }
    const float tol0 = 1.4210854715202004e-14f * (float)hes;
#pragma unroll 1
    while (true) {
        const uint32_t want = __ballot_sync(kFull, active);
        if (!want) break;
        float f[3];
        tile_f_df<n>(X, tab, want, rp, xp, f);
        if (!active) continue;
        ++fin;
        const float C00 = J[4] * J[8] - J[5] * J[7], C01 = J[5] * J[6] - J[3] * J[8], C02 = J[3] * J[7] - J[4] * J[6];
        const float C10 = J[2] * J[7] - J[1] * J[8], C11 = J[0] * J[8] - J[2] * J[6], C12 = J[1] * J[6] - J[0] * J[7];
        const float C20 = J[1] * J[5] - J[2] * J[4], C21 = J[2] * J[3] - J[0] * J[5], C22 = J[0] * J[4] - J[1] * J[3];
        const float det = J[0] * C00 + J[1] * C01 + J[2] * C02;
        const float id = -1.0f / det;
        const float d[3] = {(C00 * f[0] + C10 * f[1] + C20 * f[2]) * id, (C01 * f[0] + C11 * f[1] + C21 * f[2]) * id,
                            (C02 * f[0] + C12 * f[1] + C22 * f[2]) * id};
        const float dn = fmaxf(fabsf(d[0]), fmaxf(fabsf(d[1]), fabsf(d[2])));
        bool end = false;
        if (!edge) {
            // the FP32 phase left r within ~1e-5 of the solution: a larger step
            // or a singular J is a case for the full FP64 Newton
            if (!(dn <= 0.25f * (1.0f - kEdge))) fin = A.refine;
            // 2^-46 h_e ||J^-1||_inf: see chord_tol_df
            const float rows = fmaxf(fabsf(C00) + fabsf(C10) + fabsf(C20),
                                     fmaxf(fabsf(C01) + fabsf(C11) + fabsf(C21), fabsf(C02) + fabsf(C12) + fabsf(C22)));
            const float ct = fmaxf((float)Lim<double>::chord, tol0 * rows * fabsf(id));
            res2 = -1.0;
            if (dn <= ct) {                               // confirmed: r is kept with its own residual
                end = true;
            } else if (dn <= (float)kConfirm && dn <= (float)kTake * ct) {
                // taken; on the linear model the residual there is zero
                double g[3];
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    g[a] = fma(widen(J[3 * a]), widen(d[0]),
                               fma(widen(J[3 * a + 1]), widen(d[1]), fma(widen(J[3 * a + 2]), widen(d[2]), widen(f[a]))));
                const float e[3] = {(float)g[0], (float)g[1], (float)g[2]};
                const float c[3] = {(C00 * e[0] + C10 * e[1] + C20 * e[2]) * id, (C01 * e[0] + C11 * e[1] + C21 * e[2]) * id,
                                    (C02 * e[0] + C12 * e[1] + C22 * e[2]) * id};
#pragma unroll
                for (int a = 0; a < 3; ++a) r[a] = (widen(rp[a].hi) + widen(rp[a].lo)) + (widen(d[a]) + widen(c[a]));
                res2 = 0.0;
                fate = 2;
                active = false;
                continue;
            } else if (fin < A.refine) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {             // r + d: error-free sum, then the low parts
                    const float s = __fadd_rn(rp[a].hi, d[a]), b = __fsub_rn(s, rp[a].hi);
                    const float lo = __fadd_rn(rp[a].lo, __fadd_rn(__fsub_rn(rp[a].hi, __fsub_rn(s, b)), __fsub_rn(d[a], b)));
                    rp[a] = {s, lo};
                    df_norm(rp[a]);
                }
            }
        } else if constexpr (EDGE) {
            // on or near a bound: active set and cuts decided on r in FP64
            double rd[3], to[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) rd[a] = (double)rp[a].hi + (double)rp[a].lo;
            end = f[0] == 0.0f && f[1] == 0.0f && f[2] == 0.0f;      // exact hit
            if (!end) {
                const int on = on_bounds(rd);
                float db[3];
                end = gn_tile<float>(J, f, on, db) == 0;             // KKT point at a vertex
                double dd[3] = {(double)db[0], (double)db[1], (double)db[2]};
                const double fd[3] = {(double)f[0], (double)f[1], (double)f[2]};
                const bool small = fmaxf(fabsf(db[0]), fmaxf(fabsf(db[1]), fabsf(db[2]))) <= (float)kConfirm;
                double Jd[9];
                if (!end && small) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) Jd[k] = (double)J[k];
                    end = gn_tile<double>(Jd, fd, on, dd) == 0;
                }
                if (!end) {
                    res2 = -1.0;
                    box_tile<double>(rd, dd, to);
                    if (small) {
                        const double s[3] = {to[0] - rd[0], to[1] - rd[1], to[2] - rd[2]};
                        const double sm = fmax(fabs(s[0]), fmax(fabs(s[1]), fabs(s[2])));
                        const double ct = fmax(Lim<double>::chord, 1.4210854715202004e-14 * hes * (double)inv_norm<float>(J));
                        end = sm <= ct;
                        if (!end && sm <= kTake * ct) {   // taken on the linear model f + J s
                            double gsum = 0.0;
#pragma unroll
                            for (int a = 0; a < 3; ++a) {
                                const double g = fd[a] + Jd[3 * a] * s[0] + Jd[3 * a + 1] * s[1] + Jd[3 * a + 2] * s[2];
                                gsum += g * g;
                            }
                            res2 = gsum;
                            r[0] = to[0]; r[1] = to[1]; r[2] = to[2];
                            fate = 2;
                            active = false;
                            continue;
                        }
                    }
                    if (!end)
#pragma unroll
                        for (int a = 0; a < 3; ++a) rp[a] = df_split(to[a]);
                }
            }
        }
        if (end) {
            const double fd[3] = {(double)f[0], (double)f[1], (double)f[2]};
            res2 = fd[0] * fd[0] + fd[1] * fd[1] + fd[2] * fd[2];
            fate = 2;
        }
        if (end || fin >= A.refine) {
            active = false;
#pragma unroll
            for (int a = 0; a < 3; ++a) r[a] = (double)rp[a].hi + (double)rp[a].lo;
        }
    }
}

// What a launch of the tile kernel runs.  The mixed form is one kernel where
// the launches count (few pairs) and two where the instruction cache does:
// the loops of both phases together exceed an SM's instruction cache, and
// with 14 warps at different places in them the fetches ran at 97 % of the
// GPC cache's rate.  TILE_FINAL also runs the listed pairs (paused in the
// FP32 phase, or on a bound: a few in a hundred) from that phase to the end,
// in its first A.list_blocks blocks, beside the final steps of all others.
enum { TILE_FP64 = 0, TILE_MIXED = 1, TILE_PHASE32 = 2, TILE_FINAL = 3 };

// resident warps: the mixed kernels are capped at 128 registers (16 warps an
// SM), the FP64 one at 168 (12 warps); in blocks of 128 threads shared memory
// leaves 12 and 8 at n = 9, 8 and 8 at n = 10
template <int KIND>
struct TileLB {
    static constexpr int threads = 128;
    static constexpr int blocks = KIND == TILE_FP64 ? 3 : 4;
};

template <int n, int KIND>
struct TileSmem {
    static constexpr int v = KIND == TILE_FP64      ? Sm64<n>::BYTES
                             : KIND == TILE_PHASE32 ? Sm32<n>::BYTES
                             : Sm32<n>::BYTES > SmDf<n>::BYTES ? Sm32<n>::BYTES : SmDf<n>::BYTES;
    static constexpr int bytes = (v + 15) / 16 * 16;
};

// residual marks of unfinished pairs, and of listed pairs that only need the final steps
constexpr double kLeftOver = -1.0;     // for the full FP64 Newton
constexpr double kToFinal = -2.0;      // for the final steps
constexpr double kListed = -3.0;       // on the list
constexpr double kRhoFinal = -1.0;     // pstate.x of a listed pair that ended the FP32 phase

// one warp's rows: pairs s0..s1 of the range (listed: entries of the pause list)
template <int n, int KIND, bool FLY>
__device__ __forceinline__ void tile_rows_run(TileCtx<n, FLY>& X, const NewtonArgs& A, const BasisTab& tab, bool listed,
                                              int32_t* pl, int32_t* fbl, int64_t fbc, int64_t s0, int64_t s1)
{
    const int lane = threadIdx.x & 31;
    // rows past the end repeat the last pair and want nothing
    bool active = s0 + lane < s1;
    int64_t w = active ? s0 + lane : s1 - 1;
    int32_t q;
    if (listed) {
        w = pl[w];
        q = listed_pair(A, w);
    } else {
        q = A.order[w];
        w = result_slot(A, w, q);
        if constexpr (KIND == TILE_FINAL) {
            active = active && A.pres[w] == kToFinal;
            if (!__ballot_sync(kFull, active)) return;
        }
    }
    const int e = A.pair_elem[q] - A.ebase;
    const int64_t p = pair_point(A.pair_pt[q]);
    const int eprev = __shfl_up_sync(kFull, e, 1);
    X.e = e;
    X.heads = __ballot_sync(kFull, lane == 0 || e != eprev);
    const ElemBox& bx = A.boxes[e];
    X.bx = &bx;
    const double xs[3] = {A.pts[p], A.pts[A.P + p], A.pts[2 * A.P + p]};
    const double xc[3] = {xs[0] - bx.c[0], xs[1] - bx.c[1], xs[2] - bx.c[2]};
    const double scale = bx.scale, inv = 1.0 / scale;     // a power of two: exact
    const double xl[3] = {xc[0] * inv, xc[1] * inv, xc[2] * inv}, hes = bx.he * inv;
    double r[3], res2 = -1.0;
    float J[9];
    int fate = 3;
    bool final = false;
    NewtonState st{1.0, 0, 0, false};
    if (listed) {
        const double2 sv = A.pstate[w];
        const int code = (int)sv.y;
        st = NewtonState{sv.x, code & 3, code >> 3, false, (code & 4) != 0};
    }
    if (listed || KIND == TILE_FINAL) {
#pragma unroll
        for (int a = 0; a < 3; ++a) r[a] = A.prst[a * A.cap + w];
    }
    if constexpr (KIND == TILE_FINAL) {
        final = active && (!listed || st.rho < 0.0);
        if (final)
#pragma unroll
            for (int k = 0; k < 9; ++k) J[k] = A.jst[k * A.cap + w];
    }
    uint32_t scans = 0;
    if (KIND != TILE_FINAL && !listed) {
        bool scan = false;
        if (!warm_seed(A, p, e, r)) {
            scan = !((float)bx.dev <= kAffineSeed);
            affine_seed(bx, xc, r);
        }
        scans = __ballot_sync(kFull, active && scan);
    }
    if constexpr (KIND == TILE_FP64) {
        if (scans) tile_seed_nearest<n, double>(A.coords, A.E, scans, e, xs, tab.xi, r);
        const double xmax = fmax(fabs(xs[0]), fmax(fabs(xs[1]), fabs(xs[2]))) * inv;
        tile_solve_f64<n>(X, A, tab, active, xl, xmax, r, res2, st);
    } else {
        if (KIND != TILE_FINAL && scans) {
            const float x32[3] = {(float)xc[0], (float)xc[1], (float)xc[2]};
            float rs[3] = {(float)r[0], (float)r[1], (float)r[2]};
            tile_seed_nearest<n, float>(A.coords32, A.E, scans, e, x32, tab.xif, rs);
            r[0] = rs[0]; r[1] = rs[1]; r[2] = rs[2];
        }
        if (KIND != TILE_FINAL || listed) {
            const bool f = tile_phase32<n>(X, A, tab, active && !final, xl, hes, r, J, res2, fate, st);
            final = final || f;
        }
        if (KIND == TILE_MIXED || (KIND == TILE_FINAL && listed)) tile_final<n, true>(X, A, tab, final, xl, hes, r, J, res2, fate);
        else if (KIND == TILE_FINAL) tile_final<n, false>(X, A, tab, final, xl, hes, r, J, res2, fate);
    }
    bool put = st.paused;
    if constexpr (KIND == TILE_PHASE32) {
        if (active && final && fmax(fabs(r[0]), fmax(fabs(r[1]), fabs(r[2]))) >= (double)kEdge) {
            st.rho = kRhoFinal;
            put = true;
        }
    }
    if (KIND == TILE_PHASE32 || (KIND == TILE_FP64 && !listed)) {
        const uint32_t puts = __ballot_sync(kFull, put);
        int base = 0;
        if (puts && lane == 0) base = atomicAdd(A.pause_count, __popc(puts));
        base = __shfl_sync(kFull, base, 0);
        if (put) {
            A.pstate[w] = make_double2(st.rho, (double)(st.chord_fail + (st.flat ? 4 : 0) + 8 * st.it));
            pl[base + __popc(puts & ((1u << lane) - 1u))] = (int32_t)w;
        }
    }
    if (active) {
        A.prst[w] = r[0];
        A.prst[A.cap + w] = r[1];
        A.prst[2 * A.cap + w] = r[2];
        if (KIND == TILE_PHASE32 && final) {
#pragma unroll
            for (int k = 0; k < 9; ++k) A.jst[k * A.cap + w] = J[k];
        }
        if (put) {
            A.pres[w] = kListed;
        } else if (KIND == TILE_PHASE32 && final) {
            A.pres[w] = kToFinal;
        } else {
            A.pres[w] = res2 < 0.0 ? kLeftOver : sqrt(res2) * scale;
            if (KIND != TILE_FP64) {
                if (A.stats) atomicAdd(A.stats + fate, 1ULL);
                if (res2 < 0.0) {
                    const int32_t k = atomicAdd(A.fb_count, 1);
                    if (k < fbc) fbl[k] = (int32_t)w;
                }
            }
        }
    }
}

// Listed rows lie in as many elements: a short list is spread over a wave of
// blocks (A.list_spread, one an SM: the chain of a warp grows with its rows;
// 100,000 points in 4,096 elements, N = 7, 430 us; 490 with at least 16 rows a
// warp, 570 with 32), a long one takes 32 rows a warp, whose FP64 steps cost
// the same for any number (a batch of 24 problems 6,040 us with its lists
// spread over all list blocks, 5,550 us so).
// FLY: no stored digits (A.digits null); the launch's shared memory then ends
// with the derivative table of the mixed form
template <int n, int KIND, bool FLY = false>
__global__ void __launch_bounds__(TileLB<KIND>::threads, TileLB<KIND>::blocks) k_newton_tile(NewtonArgs A, BasisTab tab)
{
    extern __shared__ uint4 tile_sm[];
    const PairRange R = pair_range(A);
    int32_t* fbl = A.fb_list + (A.s_lo ? R.s0 : 0);
    const int64_t fbc = A.s_lo ? R.s1 - R.s0 : A.fb_cap;
    int32_t* pl = A.pause_list + (A.s_lo ? R.s0 : 0);
    TileCtx<n, FLY> X;
    if constexpr (FLY) {
        X.src = {A.coords, A.coords32, A.boxes, A.E, nullptr};
        if constexpr (KIND == TILE_MIXED) {
            float* der = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(tile_sm) + (blockDim.x >> 5) * TileSmem<n, KIND>::bytes);
            derivative_table<n>(tab, der);
            __syncthreads();
            X.src.der = der;
        }
    }
    X.sm = reinterpret_cast<unsigned char*>(tile_sm) + (threadIdx.x >> 5) * TileSmem<n, KIND>::bytes;
    X.dig = A.digits;
    const int nl = KIND == TILE_FINAL ? A.list_blocks : 0;
    // rows a warp: given, or the count spread over the warps
    auto rows_of = [&](int64_t count, int blocks, int given) {
        const int64_t nw = (int64_t)blocks * (blockDim.x >> 5), k = (count + nw - 1) / nw;
        return given > 0 ? given : (int)(k < 1 ? 1 : k > kTileRows ? kTileRows : k);
    };
    if (KIND == TILE_FINAL && (int)blockIdx.x < nl) {
        const PairRange L{0, (int64_t)*A.pause_count};
        for_each_rows(A, L, rows_of(L.s1, min(nl, A.list_spread), 0), false, (int)blockIdx.x, nl, [&](int64_t s0, int64_t s1) {
            tile_rows_run<n, KIND, FLY>(X, A, tab, true, pl, fbl, fbc, s0, s1);
        });
        return;
    }
    const bool listed = KIND == TILE_FP64 && A.resume;
    const PairRange L = listed ? PairRange{0, (int64_t)*A.pause_count} : R;
    const int nb = (int)gridDim.x - nl;
    for_each_rows(A, L, rows_of(L.s1 - L.s0, nb, listed ? 0 : A.rows), A.queue != nullptr, (int)blockIdx.x - nl, nb,
                  [&](int64_t s0, int64_t s1) {
                      tile_rows_run<n, KIND, FLY>(X, A, tab, KIND == TILE_FP64 && listed, pl, fbl, fbc, s0, s1);
                  });
}

// ---- set-up: the digits, scales and affine deviation of every element ----
// One block per element.  Shared memory: the scaled node offsets in FP64 and,
// mixed form, in FP32 and one direction's derivative values; planes of constant
// k are PL apart so that the fragments' reads of one column per k fall into
// distinct banks.  The derivative of the nodal values is taken in the
// precision its digits hold.
template <int n, bool MIXED>
struct DigitsSm {
    static constexpr int PL = n * n + (40 - n * n % 32) % 32, V = 3 * n * PL;
    static constexpr int bytes = V * (int)(sizeof(double) + (MIXED ? 2 * sizeof(float) : 0)) + (MIXED ? n * n * (int)sizeof(float) : 0);
};

// exponent of a magnitude, so that v < 2^(exponent - 1022); integer maxima of
// these take one instruction a warp, FP64 ones a pass over its pipe each
__device__ __forceinline__ int expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int expo(float v) { const int e = (__float_as_int(v) >> 23) & 0xff; return e ? e + 896 : 0; }

// k with 2^k > 2 |v| where expo(v) <= e, at least `least` (that also for e = 0)
__device__ __forceinline__ int scale_exp(int e, int least) { return min(1000, max(e > 0 ? e - 1021 : least, least)); }

template <int n, bool MIXED>
__global__ void __launch_bounds__(128) k_digits(int64_t E, const double* __restrict__ coords, ElemBox* boxes,
                                                unsigned char* __restrict__ dig, BasisTab tab)
{
    using D = TileDim<n>;
    using TB = TileBytes<n, MIXED>;
    using L = DigitsSm<n, MIXED>;
    constexpr int n3 = n * n * n, PL = L::PL;
    extern __shared__ double digits_sm[];
    double* V = digits_sm;
    float* W = reinterpret_cast<float*>(V + L::V);        // (mixed form)
    float* Vj = W + L::V;
    float* der = Vj + L::V;                               // der[i n + m] = h_m'(xi_i)
    __shared__ int4 red[4];
    const int64_t e = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (MIXED) derivative_table<n>(tab, der);
    // the largest of four values over the block, none negative
    auto block_max = [&](int4 v) {
        v = make_int4(__reduce_max_sync(kFull, v.x), __reduce_max_sync(kFull, v.y), __reduce_max_sync(kFull, v.z),
                      __reduce_max_sync(kFull, v.w));
        __syncthreads();
        if (lane == 0) red[warp] = v;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int4 o = red[w];
            v = make_int4(max(v.x, o.x), max(v.y, o.y), max(v.z, o.z), max(v.w, o.w));
        }
        return v;
    };
    int4 most = make_int4(0, 0, 0, 0);                    // exponents per coordinate; the deviation's bits
    {
        double c[3];
        float Ai[9];
#pragma unroll
        for (int a = 0; a < 3; ++a) c[a] = boxes[e].c[a];
#pragma unroll
        for (int k = 0; k < 9; ++k) Ai[k] = (float)boxes[e].Ai[k];
        for (int q = threadIdx.x; q < n3; q += 128) {
            double v[3];
            float vf[3];
            const int id[3] = {q % n, (q / n) % n, q / (n * n)}, at = q % (n * n) + PL * id[2];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                v[a] = coords[((int64_t)a * E + e) * n3 + q] - c[a];
                V[a * n * PL + at] = v[a];
                vf[a] = (float)v[a];
            }
            most = make_int4(max(most.x, expo(v[0])), max(most.y, expo(v[1])), max(most.z, expo(v[2])), most.w);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                most.w = max(most.w, __float_as_int(fabsf(Ai[3 * a] * vf[0] + Ai[3 * a + 1] * vf[1] + Ai[3 * a + 2] * vf[2] -
                                                         tab.xif[id[a]])));
        }
    }
    most = block_max(most);
    const float dev = __int_as_float(most.w);
    const int all = max(most.x, max(most.y, most.z)), ex = all > 0 ? scale_exp(all, -1000) : 0;
    // not below 2^-100 of the largest: within FP32's range
    const int3 ea = make_int3(scale_exp(most.x, ex - 100), scale_exp(most.y, ex - 100), scale_exp(most.z, ex - 100));
    for (int i = threadIdx.x; MIXED && i < L::V; i += 128) {   // (the padding too: never read back)
        const int a = i / (n * PL);
        Vj[i] = (float)(V[i] * ldexp(1.0, -(a == 0 ? ea.x : a == 1 ? ea.y : ea.z)));
    }
    __syncthreads();
    // digits of the values val[], each coordinate divided by its power of two;
    // FP64 values give 6, of which SD are kept
    auto frags = [&](auto* val, int3 sa, unsigned char* out, auto digits) {
        constexpr int SD = decltype(digits)::value;
        using TV = std::remove_pointer_t<decltype(val)>;
        for (int f = warp; f < D::KC * D::NT; f += 4) {
            const int kc = f / D::NT, t = f % D::NT, g = lane >> 2, q = lane & 3;
            const int col = 8 * t + g;                    // column a n + k is plane a n + k
            const int x = col < n ? sa.x : col < 2 * n ? sa.y : sa.z;
            RightFrag<SD> R;
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                TV v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int kap = 16 * kc + 8 * hf + 2 * q + u;
                    v[u] = kap < D::n2 && col < 3 * n ? val[col * PL + kap] : TV(0);
                }
                uint32_t d[sizeof(TV) == 8 ? 6 : 3];
                if constexpr (sizeof(TV) == 8) fields6(fixed60(v[0], x), fixed60(v[1], x), d);
                else digits2(ldexpf(v[0], -x), 1.0f, ldexpf(v[1], -x), 1.0f, d);
#pragma unroll
                for (int s = 0; s < SD; ++s) R.b[s][hf] = d[s];
            }
            R.store(out + (int64_t)f * FragBytes<SD>::v);
        }
    };
    unsigned char* out = dig + e * TB::v;                 // (dig null: scales and deviation only)
    if (dig) frags(V, ea, out, std::integral_constant<int, TB::SX>());
    // mixed form: dx/dr and dx/ds, each coordinate with its own power of two
#pragma unroll 1
    for (int m = 0; MIXED && m < 2; ++m) {
        most = make_int4(0, 0, 0, 0);
        for (int i = threadIdx.x; i < 3 * n3; i += 128) {
            const int c = i / (n * n), q = i % (n * n), at = m == 0 ? q % n : q / n, st = m == 0 ? 1 : n;
            const float w = nodal_derivative<n>(der, Vj + c * PL + q - at * st, at, st);
            W[c * PL + q] = w;
            const int x = expo(w);
            if (i < n3) most.x = max(most.x, x);
            else if (i < 2 * n3) most.y = max(most.y, x);
            else most.z = max(most.z, x);
        }
        most = block_max(most);
        const int3 sa = make_int3(scale_exp(most.x, -100), scale_exp(most.y, -100), scale_exp(most.z, -100));
        if (dig) frags(W, sa, out + TB::jac + m * TB::one, std::integral_constant<int, 3>());
        if (threadIdx.x == 0) {
            boxes[e].jscale[m][0] = ldexpf(1.0f, sa.x + ea.x - ex);
            boxes[e].jscale[m][1] = ldexpf(1.0f, sa.y + ea.y - ex);
            boxes[e].jscale[m][2] = ldexpf(1.0f, sa.z + ea.z - ex);
        }
        __syncthreads();                                  // W is rewritten
    }
    if (threadIdx.x == 0) {
        boxes[e].scale = ldexp(1.0, ex);
        boxes[e].dev = dev;
        boxes[e].cscale[0] = ldexpf(1.0f, ea.x - ex);
        boxes[e].cscale[1] = ldexpf(1.0f, ea.y - ex);
        boxes[e].cscale[2] = ldexpf(1.0f, ea.z - ex);
    }
}

}  // namespace fpg
