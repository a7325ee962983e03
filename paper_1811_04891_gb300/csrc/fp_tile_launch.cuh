// fp_tile_launch.cuh -- how the tile kernels (fp_tile.cuh) of one order are
// launched: row and block counts, the two-launch sequence, and the digits.
#pragma once
#include <algorithm>
#include <atomic>

#include "fp_tile.cuh"

namespace fpg {

static int sm_count()
{
    static std::atomic<int> known{0};
    if (const int v = known.load()) return v;
    int dev = 0, k = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&k, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || k < 1)
        return 152;
    known.store(k);
    return k;
}

// a kernel's dynamic shared memory limit, raised once per device
template <typename K>
static cudaError_t raise_smem(std::atomic<uint64_t>& done, K kernel, int bytes)
{
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
    if (done.load() & bit) return cudaSuccess;
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (err == cudaSuccess) done.fetch_or(bit);
    return err;
}

// (tile kernels: blocks of up to four warps)
template <int n, int KIND, bool FLY>
constexpr int tile_smem(int warps) { return warps * TileSmem<n, KIND>::bytes + (FLY && KIND == TILE_MIXED ? n * n * (int)sizeof(float) : 0); }

template <int n, int KIND, bool FLY = false>
static cudaError_t tile_prepare()
{
    static std::atomic<uint64_t> done{0};
    return raise_smem(done, k_newton_tile<n, KIND, FLY>, tile_smem<n, KIND, FLY>(4));
}

// blocks of `block` threads that fit one SM at once (asked of the runtime once per form and block size)
template <int n, int KIND, bool FLY = false>
static int tile_fit(int block)
{
    static std::atomic<int> known[5];
    std::atomic<int>& slot = known[std::min(block / 32, 4)];
    if (const int v = slot.load()) return v;
    int k = 0;
    cudaError_t e = tile_prepare<n, KIND, FLY>();
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_newton_tile<n, KIND, FLY>, block,
                                                          (size_t)tile_smem<n, KIND, FLY>(block / 32));
    if (e != cudaSuccess || k < 1) return 1;
    slot.store(k);
    return k;
}

// grid: 0 = one warp per na.rows pairs of npairs; persistent (npairs < 0) =
// every block that fits the GPU at once; otherwise as given
template <int n, int KIND, bool FLY = false>
static cudaError_t launch_tile(const NewtonArgs& na, const BasisTab& tab, int64_t npairs, int block, unsigned grid,
                               cudaStream_t s)
{
    // whole warps, at most the four of the launch bounds: each has its own shared memory
    if (block < 32 || block > TileLB<KIND>::threads || block % 32 != 0) return cudaErrorInvalidValue;
    const int per = block / 32;
    const cudaError_t err = tile_prepare<n, KIND, FLY>();
    if (err != cudaSuccess) return err;
    if (npairs < 0) grid = (unsigned)(sm_count() * tile_fit<n, KIND, FLY>(block));
    else if (grid == 0) grid = (unsigned)std::max<int64_t>(1, (npairs + (int64_t)per * na.rows - 1) / ((int64_t)per * na.rows));
    grid += na.list_blocks;
    k_newton_tile<n, KIND, FLY><<<grid, block, (size_t)tile_smem<n, KIND, FLY>(per), s>>>(na, tab);
    count_launch();
    return cudaGetLastError();
}

// Tile kernels: evaluations of a pair in the first pass.  Most pairs take
// two evaluations of the map with its Jacobian (and then chord or final
// steps); the few that need more (border points, candidates the point lies
// outside of) would keep their warps' other rows waiting, so they are listed
// and continued by a second launch, dense again.
// The mixed form's two phases are then launches of their own as well: either
// one's code fits the instruction cache, both together do not (one kernel was
// 30 % slower).  With few pairs one launch is shorter: N = 7, 20,000 points in
// 4,096 elements, 277 against 307 us; 100,000 points 450 against 430.
constexpr int kTilePassMixed = 3;
constexpr int kTilePass = 3;
constexpr int64_t kTwoPass = 65536;

// Rows per warp of the tile kernels when the pair count is known: 32 gives
// every lane a row; with few pairs, only as many as it takes to fill the GPU
// once (or a whole number of times): the time is then that of one warp's
// chain over its elements' fragments.  N = 7, 20,000 points in 4,096
// elements: 8 rows 1.3 waves 333 us, 10 rows one wave 277 us; 3,000 points:
// 4 rows 208 us, 2 rows 183 us.
static int tile_rows(int64_t npairs, int warps)
{
    if (npairs >= kTwoPass) return 32;
    const int64_t all = (int64_t)sm_count() * warps, waves = (npairs + 32 * all - 1) / (32 * all);
    const int64_t k = (npairs + all * waves - 1) / (all * waves);
    return (int)(k < 1 ? 1 : k);
}

// Few pairs (a launch of fewer than two blocks per SM at `block` threads):
// smaller blocks, down to one warp, so that every SM gets work.  The block
// size changes only the schedule, not any pair's result.  Blocks stay whole
// warps (any multiple of 32 may be asked for: 96 goes to 32, not to 48): the
// tile kernels' warps share no rows and every lane of a warp takes part.
constexpr int halved_block(int block) { return block / 2 / 32 * 32 < 32 ? 32 : block / 2 / 32 * 32; }

constexpr bool halves_to_whole_warps()
{
    for (int b = 32; b <= 1024; b += 32)
        for (int h = b; h > 32; h = halved_block(h))
            if (halved_block(h) % 32 != 0 || halved_block(h) < 32 || halved_block(h) >= h) return false;
    return true;
}
static_assert(halves_to_whole_warps(), "spread_block: whole warps only");

static int spread_block(int64_t npairs, int block)
{
    const int nsm = sm_count();
    while (block > 32 && (npairs + block - 1) / block < 2 * nsm) block = halved_block(block);
    return block;
}

// The Newton launches of a tile order (na: see newton_form); grid == 0: sized
// from npairs, or persistent when the caller gave persistent_blocks.
template <int n, bool MIXED>
static cudaError_t newton_tile(const FindArgs& a, NewtonArgs na, int64_t npairs, const BasisTab& tab, int block,
                               unsigned grid, cudaStream_t s)
{
    cudaError_t err;
    constexpr int KIND = MIXED ? TILE_MIXED : TILE_FP64;
    int tblock = std::min(block, 128);               // threads per block the tile kernels are built for
    const bool fixed = a.persistent_blocks > 0 || a.queue;
    int64_t launch = npairs;                         // < 0: a persistent grid
    if (!fixed) {
        na.rows = tile_rows(npairs, tblock / 32 * (na.digits ? tile_fit<n, KIND>(tblock) : tile_fit<n, KIND, true>(tblock)));
        tblock = spread_block(npairs * 32 / na.rows, tblock);
        grid = 0;
    } else {
        na.rows = a.queue ? 32 : 0;
        if (grid == 0) launch = -1;
    }
    // two passes (and the mixed form's phases in launches of their own)
    // when the pairs fill the GPU several times over
    const bool two = na.digits && a.pstate && a.pause_list && (a.jst || !MIXED) && npairs >= kTwoPass;
    na.first_pass = 0x7fffffff;
    if (!na.digits) {                                // no stored digits: one launch that makes them
        err = launch_tile<n, KIND, true>(na, tab, launch, tblock, grid, s);
    } else if (!two) {
        err = launch_tile<n, KIND>(na, tab, launch, tblock, grid, s);
    } else {
        na.pstate = a.pstate;
        na.jst = a.jst;
        na.pause_list = a.pause_list;
        na.pause_count = a.s_lo ? a.pause_count : a.scan_tmp + 1;
        if ((err = cudaMemsetAsync(na.pause_count, 0, sizeof(int32_t), s)) != cudaSuccess) return err;
        NewtonArgs nr = na;                          // the paused solves
        nr.resume = true;
        nr.queue = nullptr;
        nr.rows = 0;
        na.first_pass = MIXED ? kTilePassMixed : kTilePass;
        if constexpr (MIXED) {
            err = launch_tile<n, TILE_PHASE32>(na, tab, launch, tblock, grid, s);
            if (err == cudaSuccess && a.queue) err = cudaMemsetAsync(a.queue, 0, sizeof(int32_t), s);
            // blocks for a list of one pair in twelve at 32 rows a warp (longer ones loop)
            na.first_pass = 0x7fffffff;
            na.list_blocks = (int)std::max<int64_t>(sm_count(), npairs / (12 * tblock));
            na.list_spread = sm_count();
            if (err == cudaSuccess) err = launch_tile<n, TILE_FINAL>(na, tab, launch, tblock, grid, s);
        } else {
            err = launch_tile<n, TILE_FP64>(na, tab, launch, tblock, grid, s);
            if (err == cudaSuccess) err = launch_tile<n, TILE_FP64>(nr, tab, -1, tblock, 0, s);
        }
    }
    return err;
}

template <int n, bool MIXED>
static cudaError_t digits_form(int64_t E, const double* coords, ElemBox* boxes, unsigned char* dig, const BasisTab& tab,
                               cudaStream_t s)
{
    constexpr int smem = DigitsSm<n, MIXED>::bytes;
    static std::atomic<uint64_t> done{0};
    const cudaError_t err = raise_smem(done, k_digits<n, MIXED>, smem);
    if (err != cudaSuccess) return err;
    k_digits<n, MIXED><<<(unsigned)E, 128, smem, s>>>(E, coords, boxes, dig, tab);
    count_launch();
    return cudaGetLastError();
}

}  // namespace fpg
