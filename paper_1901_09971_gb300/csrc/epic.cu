// EPIC interpolation of the sparse flow into a dense field (Section 2,
// "Interpolation": an affine model fitted to the k nearest sparse vectors under a
// geodesic distance that penalises crossing image edges, the edges taken from
// image gradients; Section 3 "Parameters": k = 128). The paper gives no formulas;
// the reading, with every distance an exact integer, is stated with
// epic_interpolate in degraf.h.
//
// Launches on the caller's stream:
//   1. edge cost C = base + gain (|Gx| + |Gy|) per pixel (integer Sobel), labels and the
//      call's counters cleared;
//   2. seeds claim their pixels (atomicMin on (distance 0, index)), then keep a
//      pixel only where they hold it;
//   3. geodesic Voronoi labelling by tile-local relaxation: 32 x 32 tiles iterate
//      min-plus updates of the (distance, seed) keys in registers until they are
//      locally stable, write improvements back and count them; one cooperative launch
//      repeats passes until one changes nothing. Relaxation converges to the unique
//      fixed point, the lexicographic (distance, seed) minimum, whatever the order;
//   4-6. seed graph: links of 4-adjacent pixels in different cells are counted,
//      scanned into offsets (three launches: block scans, a scan of the block
//      totals, the block offsets added) and filled into per-seed lists;
//   7-8. each list keeps one link per neighbour (its smallest weight), in a 16-byte
//      record with the neighbour's own smallest weight, so a search discovers a seed
//      with one load;
//   9. per seed, one warp runs Dijkstra over the seed graph with batch settling
//      (every frontier seed within its smallest incoming link of the frontier
//      minimum is final, so about 14 steps settle the 128 nearest instead of 128
//      pops), a hash of discovered seeds in shared memory, then sorts the settled
//      (distance, index) keys and sums the weighted affine fit's terms over the first k
//      (double-float); a thread per seed solves the fits (FP64). A search that outgrows
//      the hash (384 seeds;
//      1024 for k > 160) or the sort buffer (256; 512) is queued and redone by a
//      retry kernel with room for 8192;
//   10. dense flow: every pixel evaluates its seed's model; a failure of the call goes into
//      the library's status word.
// Clears and the report in kernels that run anyway instead of two memsets and a launch:
// 138 -> 131 us on the 256x128 pair.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace {

constexpr unsigned long long kNone = ~0ull;
constexpr int kIdxBits = 24;
constexpr unsigned long long kIdxMask = (1ull << kIdxBits) - 1;
constexpr long long kDistLimit = 1ll << 40;  // the distance field of a packed key
constexpr int kTile = 32, kBand = 4;         // Voronoi tiles: 32 x 32 pixels, 32 x 8 threads, four rows a warp
constexpr int kMaxPasses = 4096;
constexpr int kThreads = 256;

// Distances on the frame fit 31 bits: at most W + H steps of at most twice the largest
// pixel cost (base 4096, gain 32, Sobel magnitudes 1020 + 1020). A link's weight, two
// distances and a step, fits 32.
constexpr long long kMaxStep = 2ll * (4096 + 32 * 2040);
static_assert(DGF_EPIC_MAX_W_PLUS_H * kMaxStep < (1ll << 31), "distances of 31 bits");
static_assert(2 * DGF_EPIC_MAX_W_PLUS_H * kMaxStep + kMaxStep < 0xffffffffll, "link weights of 32 bits");
constexpr unsigned kNoLink = 0xffffffffu;  // min link weight of a seed without links

// Device status bits (any of them makes the call return DGF_ERR_DEVICE).
enum : int { kErrFrontier = 1, kErrFill = 4, kErrRange = 8, kErrPasses = 16, kErrSync = 32 };
constexpr unsigned kBarrierTries = 1u << 24;  // polls (20 ns naps) before a grid barrier gives up

// The kernels of a call depend on one another in order and many take 2 to 5 us, so each
// allows the next one's launch at its start (follow) and a kernel launched with
// launch_next waits for the end of the one before it, and its writes, before it touches
// memory (begin_after). Only launch and block set-up overlap: 256x128 pair 131 -> 106 us,
// 1242x375 842 -> 817.
__device__ __forceinline__ void follow() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void begin_after()
{
    follow();
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launches a kernel that calls begin_after first. Not for kernels that read what the call
// writes by __ldg (the search): its data must not change while the kernel is resident.
// With plain loads the search gains nothing from it (107 and 815 us).
template <typename... P, typename... A>
void launch_next(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.stream = stream;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    (void)cudaLaunchKernelEx(&c, kernel, P(args)...);  // a failure is read by launch_status
}

__device__ __forceinline__ bool is_tracked(uint8_t s) { return s == DGF_TRACKED || s == DGF_MAXITER; }

__global__ void __launch_bounds__(kThreads) epic_cost_kernel(const uint8_t* img, int W, int H, int pitch, int base,
                                                             int gain, int* cost, unsigned long long* key,
                                                             int* counters, int n_counters)
{
    follow();
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
    const int id = (blockIdx.y * gridDim.x + blockIdx.x) * kThreads + threadIdx.y * 32 + threadIdx.x;
    for (int i = id; i < n_counters; i += gridDim.x * gridDim.y * kThreads) counters[i] = 0;
    if (x >= W || y >= H) return;
    const int xm = max(x - 1, 0), xp = min(x + 1, W - 1);
    const uint8_t* r0 = img + (size_t)max(y - 1, 0) * pitch;
    const uint8_t* r1 = img + (size_t)y * pitch;
    const uint8_t* r2 = img + (size_t)min(y + 1, H - 1) * pitch;
    const int a = r0[xm], b = r0[x], c = r0[xp], d = r1[xm], f = r1[xp], g = r2[xm], h = r2[x], i = r2[xp];
    const int gx = (c - a) + 2 * (f - d) + (i - g);
    const int gy = (g - a) + 2 * (h - b) + (i - c);
    const size_t o = (size_t)y * W + x;
    cost[o] = base + gain * (abs(gx) + abs(gy));
    key[o] = kNone;
}

__global__ void __launch_bounds__(kThreads) epic_seed_kernel(const float2* pts, const uint8_t* status, int n, int W,
                                                             int H, unsigned long long* key, int* seed_pix, int* cnt)
{
    begin_after();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    cnt[i] = 0;
    int o = -1;
    if (is_tracked(status[i])) {
        const float2 p = pts[i];
        // x + 1/2 is exact in FP32 below 2^22; NaN clamps to 0
        const int x = (int)fminf(fmaxf(floorf(p.x + 0.5f), 0.f), (float)(W - 1));
        const int y = (int)fminf(fmaxf(floorf(p.y + 0.5f), 0.f), (float)(H - 1));
        o = y * W + x;
        atomicMin(&key[o], (unsigned long long)i);  // distance 0: the lowest index holds the pixel
    }
    seed_pix[i] = o;
}

__global__ void __launch_bounds__(kThreads) epic_seed_owner_kernel(const unsigned long long* key, int n, int* seed_pix)
{
    begin_after();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const int o = seed_pix[i];
    if (o >= 0 && key[o] != (unsigned long long)i) seed_pix[i] = -1;
}

// Labelling keys in registers and shared memory: distance (31 bits) in the high word, seed
// in the low one, so a step adds its weight to one word. An unreached pixel holds kFar,
// from which no step improves anything. Pixels outside the frame hold 0, which nothing
// improves, and steps from them weigh kWall, which ends at kFar: no improvement either.
constexpr unsigned kWall = 0xc0000000u;
constexpr unsigned long long kFar = (unsigned long long)kWall << 32;
static_assert(kWall + kMaxStep < (1ll << 32), "a step from an unreached pixel stays in 32 bits");
__device__ __forceinline__ unsigned long long step_from(unsigned long long kn, unsigned w)
{
    return ((unsigned long long)((unsigned)(kn >> 32) + w) << 32) | (unsigned)kn;
}
__device__ __forceinline__ void relax(unsigned long long& best, unsigned long long kn, unsigned w)
{
    best = min(best, step_from(kn, w));
}

// Rows of a tile that other warps read: the first and the last of each warp's band.
// Plain 8-byte shared accesses (never torn), volatile so that every sweep reads anew.
struct VoronoiEdges {
    volatile unsigned long long top[kTile / kBand][kTile], bot[kTile / kBand][kTile];
};

// One relaxation pass over the 32 x 32 tile at (x0, y0): a warp owns a band of four rows
// and a lane a column of it, keys and edge weights in registers, the neighbouring
// tiles' border keys (halo) fixed for the pass. A sweep relaxes each pixel from its
// left and right neighbours (shuffles), then down and up the band (a path runs
// through the whole band in one sweep), the bands' border rows passing through shared
// memory. The min-plus fixed point does not depend on the order, so warps sweep
// without waiting for one another (a stale border row is a valid upper bound) and only
// every third sweep is closed by a barrier before and a vote after it: once it changes
// nothing, every pixel was checked against final neighbours. Improved keys are
// written back (the tile's pixels are written by nobody else); counts the tile in
// changed[pass] if any key improved. Called by every thread of the block. With fresh
// unset, T still holds the tile's keys and weights from the block's last pass (a block
// that owns one tile loads them once and then only the halo).
// What bounds it is the latency of one sweep times the longest path inside a tile
// (shortest paths through seedless areas wind for 50 pixels and more). With a thread
// per four scattered pixels, all keys in shared memory and two barriers a sweep, a
// sweep took about 1,250 cycles and moved a path one pixel: 227 us of labelling on the
// 1242x375 pair, about 110 us now.
struct VoronoiBand {
    unsigned long long k[kBand];
    unsigned wl[kBand], wr[kBand], wu[kBand], wd[kBand];  // weights of the steps into the lane's pixels
};
__device__ __forceinline__ void voronoi_tile(const int* cost, unsigned long long* key, int W, int H, int* changed,
                                             int pass, int x0, int y0, VoronoiEdges& E, VoronoiBand& T, bool fresh)
{
    const int lane = threadIdx.x, w = threadIdx.y;
    const int x = x0 + lane, yb = y0 + kBand * w;
    auto load_key = [&](int px, int py) {
        if (px < 0 || px >= W || py < 0 || py >= H) return 0ull;
        // halo keys belong to other tiles, which may lower them concurrently; any
        // value read is a valid upper bound
        const unsigned long long v = *reinterpret_cast<const volatile unsigned long long*>(key + (size_t)py * W + px);
        return v == kNone ? kFar : ((v >> kIdxBits) << 32) | (v & kIdxMask);
    };
    auto load_cost = [&](int px, int py) {
        return px >= 0 && px < W && py >= 0 && py < H ? (unsigned)cost[(size_t)py * W + px] : kWall;
    };
    // weight of the step into a pixel of cost a from one of cost b
    auto edge = [](unsigned a, unsigned b) { return a == kWall ? 0u : b == kWall ? kWall : a + b; };
    unsigned long long(&k)[kBand] = T.k;
    const int xs = lane == 0 ? x - 1 : x + 1;  // beside the tile, for lanes 0 and 31
    const bool outer = lane == 0 || lane == 31;
    if (fresh) {
        unsigned c[kBand + 2];
#pragma unroll
        for (int r = 0; r < kBand; ++r) k[r] = load_key(x, yb + r);
#pragma unroll
        for (int r = 0; r < kBand + 2; ++r) c[r] = load_cost(x, yb + r - 1);
#pragma unroll
        for (int r = 0; r < kBand; ++r) {
            const unsigned cs = outer ? load_cost(xs, yb + r) : 0u;
            unsigned cl = __shfl_up_sync(0xffffffffu, c[r + 1], 1), cr = __shfl_down_sync(0xffffffffu, c[r + 1], 1);
            if (lane == 0) cl = cs;
            if (lane == 31) cr = cs;
            T.wl[r] = edge(c[r + 1], cl);
            T.wr[r] = edge(c[r + 1], cr);
            T.wu[r] = edge(c[r + 1], c[r]);
            T.wd[r] = edge(c[r + 1], c[r + 2]);
        }
    }
    unsigned long long orig[kBand], side[kBand];  // side: the halo beside lanes 0 and 31
#pragma unroll
    for (int r = 0; r < kBand; ++r) {
        orig[r] = k[r];
        side[r] = outer ? load_key(xs, yb + r) : kFar;
    }
    // the halo rows above and below the tile, or the neighbouring bands' border rows
    const bool first = w == 0, last = w == kTile / kBand - 1;
    const unsigned long long above = first ? load_key(x, yb - 1) : kFar, below = last ? load_key(x, yb + kBand) : kFar;
    E.top[w][lane] = k[0];
    E.bot[w][lane] = k[kBand - 1];
    __syncthreads();
    auto sweep = [&]() {
        const unsigned long long up = first ? above : E.bot[w - 1][lane], dn = last ? below : E.top[w + 1][lane];
        bool ch = false;
        unsigned long long b[kBand];
#pragma unroll
        for (int r = 0; r < kBand; ++r) {
            unsigned long long l = __shfl_up_sync(0xffffffffu, k[r], 1), t = __shfl_down_sync(0xffffffffu, k[r], 1);
            if (lane == 0) l = side[r];
            if (lane == 31) t = side[r];
            b[r] = k[r];
            relax(b[r], l, T.wl[r]);
            relax(b[r], t, T.wr[r]);
        }
        relax(b[0], up, T.wu[0]);
#pragma unroll
        for (int r = 1; r < kBand; ++r) relax(b[r], b[r - 1], T.wu[r]);
        relax(b[kBand - 1], dn, T.wd[kBand - 1]);
#pragma unroll
        for (int r = kBand - 2; r >= 0; --r) relax(b[r], b[r + 1], T.wd[r]);
#pragma unroll
        for (int r = 0; r < kBand; ++r) {
            ch |= b[r] < k[r];
            k[r] = b[r];
        }
        E.top[w][lane] = k[0];
        E.bot[w][lane] = k[kBand - 1];
        return ch;
    };
    // a sweep between barriers extends every shortest path by at least one step, so the
    // tile is stable after at most kTile^2 rounds
    for (int it = 0; it <= kTile * kTile; ++it) {
        if (it) {
            sweep();
            sweep();
            __syncthreads();
        }
        if (!__syncthreads_or(sweep())) break;
    }
    bool improved = false;
#pragma unroll
    for (int r = 0; r < kBand; ++r)
        if (k[r] < orig[r]) {  // (never outside the frame: 0 there)
            key[(size_t)(yb + r) * W + x] = ((k[r] >> 32) << kIdxBits) | (k[r] & kIdxMask);
            improved = true;
        }
    // (also keeps the next tile's border rows behind this tile's last sweep)
    if (__syncthreads_or(improved) && lane == 0 && w == 0) atomicAdd(&changed[pass], 1);
}

// Barrier of all blocks of a cooperative launch (all co-resident): arrivals on a
// counter that grows by the grid size per use; the waits are bounded, and false
// comes back once a block gave up.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        __threadfence();  // this block's key and counter updates before its arrival
        atomicAdd(count, 1u);
        int ok = 0;
        for (unsigned i = 0; i < kBarrierTries; ++i) {
            if (*reinterpret_cast<volatile unsigned*>(count) >= target) {
                ok = 1;
                break;
            }
            __nanosleep(20);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Geodesic Voronoi labelling in one cooperative launch: every pass relaxes all tiles
// (block b takes tiles b, b + grid, ...), a grid barrier closes it, and the passes
// stop at the first that changed nothing (every block reads the same count after
// the barrier) or after kMaxPasses, which is recorded as a failure; so is a barrier
// that gave up. No host round trip between passes.
__global__ void __launch_bounds__(kThreads, 4) epic_voronoi_kernel(const int* cost, unsigned long long* key, int W, int H,
                                                                int* changed, unsigned* sync_count, int* err)
{
    __shared__ VoronoiEdges edges;
    VoronoiBand band;
    const int tiles_x = (W + kTile - 1) / kTile, n_tiles = tiles_x * ((H + kTile - 1) / kTile);
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0;
    for (int pass = 0; pass < kMaxPasses; ++pass) {
        for (int t = blockIdx.x; t < n_tiles; t += gridDim.x)
            voronoi_tile(cost, key, W, H, changed, pass, (t % tiles_x) * kTile, (t / tiles_x) * kTile, edges, band,
                         pass == 0 || n_tiles > (int)gridDim.x);
        if (!grid_barrier(sync_count, (unsigned)(pass + 1) * gridDim.x)) {
            if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(err, kErrSync);
            return;
        }
        if (*reinterpret_cast<volatile int*>(changed + pass) == 0) return;
    }
    if (lead) atomicOr(err, kErrPasses);
}

// Seed-graph links of pixel o with its right and lower neighbours.
template <bool FILL>
__global__ void __launch_bounds__(kThreads) epic_links_kernel(const unsigned long long* key, const int* cost, int W,
                                                              int H, int* cnt, const int* off, int* cur, int* adj_t,
                                                              unsigned* adj_w, int* err)
{
    begin_after();
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
    if (x >= W || y >= H) return;
    const size_t o = (size_t)y * W + x;
    const unsigned long long k = key[o];
    if (k == kNone) return;
    const int s = (int)(k & kIdxMask);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (q == 0 ? x + 1 >= W : y + 1 >= H) continue;
        const size_t o2 = q == 0 ? o + 1 : o + W;
        const unsigned long long k2 = key[o2];
        if (k2 == kNone || (int)(k2 & kIdxMask) == s) continue;
        const int t = (int)(k2 & kIdxMask);
        if (!FILL) {
            atomicAdd(&cnt[s], 1);
            atomicAdd(&cnt[t], 1);
            continue;
        }
        const unsigned w = (unsigned)(k >> kIdxBits) + (unsigned)(cost[o] + cost[o2]) + (unsigned)(k2 >> kIdxBits);
        const int ps = atomicAdd(&cur[s], 1), pt = atomicAdd(&cur[t], 1);
        if (ps < off[s + 1]) {
            adj_t[ps] = t;
            adj_w[ps] = w;
        } else {
            atomicOr(err, kErrFill);
        }
        if (pt < off[t + 1]) {
            adj_t[pt] = s;
            adj_w[pt] = w;
        } else {
            atomicOr(err, kErrFill);
        }
    }
}

// Exclusive scan of the link counts into offsets (off[n] = total) and cursors: one
// block walks the counts in coalesced tiles of 1024, carrying the running total.
__global__ void __launch_bounds__(1024) epic_scan_kernel(const int* cnt, int n, int* off, int* cur)
{
    begin_after();
    __shared__ int wsum[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int carry = 0;
    for (int base = 0; base < n; base += 1024) {
        const int i = base + t;
        const int v = i < n ? cnt[i] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int z = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, z, o);
                if (lane >= o) z += y;
            }
            wsum[lane] = z;
        }
        __syncthreads();
        const int excl = carry + (w ? wsum[w - 1] : 0) + x - v;
        if (i < n) {
            off[i] = excl;
            cur[i] = excl;
        }
        carry += wsum[31];
        __syncthreads();
    }
    if (t == 0) off[n] = carry;
}

// Multi-block exclusive scan of the link counts: each block scans 1024 counts and
// publishes its total; the one-block scan above turns the totals into block
// offsets; a last pass adds them (and fills the cursors).
__global__ void __launch_bounds__(1024) epic_scan_blocks_kernel(const int* cnt, int n, int* off, int* bsum)
{
    begin_after();
    __shared__ int wsum[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int i = blockIdx.x * 1024 + t;
    const int v = i < n ? cnt[i] : 0;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        int z = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        wsum[lane] = z;
    }
    __syncthreads();
    if (i < n) off[i] = (w ? wsum[w - 1] : 0) + x - v;
    if (t == 0) bsum[blockIdx.x] = wsum[31];
}

__global__ void __launch_bounds__(1024) epic_scan_add_kernel(const int* boff, int n, int nb, int* off, int* cur)
{
    begin_after();
    const int i = blockIdx.x * 1024 + threadIdx.x;
    if (i < n) {
        const int o = off[i] + boff[blockIdx.x];
        off[i] = o;
        cur[i] = o;
    }
    if (i == 0) off[n] = boff[nb];
}

struct KnnArgs {
    const float2* pts;
    const float2* flow;
    const int* seed_pix;
    const int* off;
    const int* end_of;
    const unsigned* minin;
    const int4* adj;  // link records: neighbour, its smallest link weight, the link's weight
    double* models;  // [n][6]
    const int* list;        // the seeds that hold a pixel, in any order
    const int* list_count;  // their number
    double* sums;           // [end - begin][12]: the fits' weighted sums, solved by epic_solve_kernel
    int begin, end;         // this launch's part of the list
    const float2* weights;  // [n_weights]: the fit weights of distances 0 .. n_weights - 1 (double-float)
    int n_weights;
    int* err;
    int* retry_count;
    int* retry_list;
    int32_t* knn_idx;
    int64_t* knn_dist;
    int32_t* knn_count;
    double* dbg_models;
    uint8_t* fit_kind;
    int n, k, model;
    double a_per_unit, min_spread2;  // kernel decay per unit of distance: a / (2 cost_base)
};

// Per-warp shared layout of one search: a hash of HCAP discovered seeds (index,
// tentative distance, smallest incoming link weight), the frontier as a list of FCAP
// hash slots, and the settled keys (SCAP, later sorted in place). Distances are of
// type DT: 32 bits in the fast layouts (half the shared traffic of 64, and a native
// shared atomic minimum where a 64-bit one is a compare-and-swap loop), 64 in the
// retry kernel's.
template <typename DT, int HCAP, int FCAP, int SCAP>
struct KnnLayout {
    static_assert(HCAP % 128 == 0 && SCAP % 32 == 0 && HCAP <= 32768, "sizes");
    static constexpr size_t o_hdist = (size_t)HCAP * 4;
    static constexpr size_t o_sort = o_hdist + (size_t)HCAP * sizeof(DT);
    static constexpr size_t o_minin = o_sort + (size_t)SCAP * 8;
    static constexpr size_t o_front = o_minin + (size_t)HCAP * 4;
    static constexpr size_t o_count = (o_front + (size_t)FCAP * 2 + 15) & ~(size_t)15;
    static constexpr size_t bytes = o_count + 16;
};

// The fast layouts hold every search of the benchmark scenes (at k = 128 at most
// about 250 discovered and 171 settled seeds, in a 384-slot hash; larger k takes
// the larger one); a search that outgrows them is redone by the retry kernel with
// room for 8192.
constexpr int kFastWarps = 4, kSmallK = 160;
using SmallLayout = KnnLayout<unsigned, 384, 256, 256>;
using LargeLayout = KnnLayout<unsigned, 1024, 512, 512>;
constexpr int kBigH = 8192, kBigF = 8192, kBigS = 8192;  // the retry kernel runs one block per SM
using RetryLayout = KnnLayout<long long, kBigH, kBigF, kBigS>;
constexpr int kRetry = 16;  // search status: capacity exceeded, redo with the large layout

// exp(-y) for y >= 0 by the table-driven method of Tang (ACM TOMS 15(2), 1989):
// y = (32 q + j) ln2 / 32 + r with |r| <= ln2 / 64, so exp(-y) = 2^-q 2^(-j/32)
// exp(-r), exp(-r) by its degree-6 Taylor polynomial (truncation below 4e-18); the
// reduction uses a two-part ln2 / 32 and fused multiply-adds; the power of two is
// built from exponent bits. Within 2 ulps of the result (measured against an
// extended-precision exp: 1.93 ulps on normal results, 1.27 on subnormal ones); 0
// from y = 745.2 on, where exp(-y) is below half the smallest subnormal.
__device__ const double kExp2Frac[32] = {  // 2^(-j/32), correctly rounded
    0x1.0000000000000p+0, 0x1.f50765b6e4540p-1, 0x1.ea4afa2a490dap-1, 0x1.dfc97337b9b5fp-1,
    0x1.d5818dcfba487p-1, 0x1.cb720dcef9069p-1, 0x1.c199bdd85529cp-1, 0x1.b7f76f2fb5e47p-1,
    0x1.ae89f995ad3adp-1, 0x1.a5503b23e255dp-1, 0x1.9c49182a3f090p-1, 0x1.93737b0cdc5e5p-1,
    0x1.8ace5422aa0dbp-1, 0x1.82589994cce13p-1, 0x1.7a11473eb0187p-1, 0x1.71f75e8ec5f74p-1,
    0x1.6a09e667f3bcdp-1, 0x1.6247eb03a5585p-1, 0x1.5ab07dd485429p-1, 0x1.5342b569d4f82p-1,
    0x1.4bfdad5362a27p-1, 0x1.44e086061892dp-1, 0x1.3dea64c123422p-1, 0x1.371a7373aa9cbp-1,
    0x1.306fe0a31b715p-1, 0x1.29e9df51fdee1p-1, 0x1.2387a6e756238p-1, 0x1.1d4873168b9aap-1,
    0x1.172b83c7d517bp-1, 0x1.11301d0125b51p-1, 0x1.0b5586cf9890fp-1, 0x1.059b0d3158574p-1,
};

__device__ __forceinline__ double exp_neg(double y)
{
    if (!(y < 745.2)) return 0.0;
    const double kf = rint(y * 0x1.71547652b82fep+5);  // y * 32 / ln2
    double r = fma(-kf, 0x1.62e42fefa39efp-6, y);      // ln2 / 32, leading part
    r = fma(-kf, 0x1.abc9e3b39803fp-61, r);            // and the rest
    const double x = -r;
    double e = 1.0 / 720.0;
    e = fma(e, x, 1.0 / 120.0);
    e = fma(e, x, 1.0 / 24.0);
    e = fma(e, x, 1.0 / 6.0);
    e = fma(e, x, 0.5);
    e = fma(e, x, 1.0);
    e = fma(e, x, 1.0);
    const int k = (int)kf, q = k >> 5;  // q <= 1075: 2^-q as two normal powers of two
    const double s1 = __longlong_as_double((long long)(1023 - (q >> 1)) << 52);
    const double s2 = __longlong_as_double((long long)(1023 - (q - (q >> 1))) << 52);
    return e * __ldg(&kExp2Frac[k & 31]) * s1 * s2;
}

// Double-float arithmetic (an unevaluated pair hi + lo of FP32 values, about 48
// significant bits; Dekker 1971, Knuth's TwoSum): the fit's per-neighbour products
// and sums run on GB300's wide FP32 pipe instead of its narrow FP64 pipe, at an
// accuracy far inside what the fit needs. Written with the _rn intrinsics so that
// no addition is contracted or reordered.
struct dfl {
    float hi, lo;
};

__device__ __forceinline__ dfl two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ dfl fast_two_sum(float a, float b)  // |a| >= |b| or a == 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ dfl df_mul(dfl a, dfl b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p)));
    return fast_two_sum(p, e);
}

__device__ __forceinline__ dfl df_mul(dfl a, float b)
{
    const float p = __fmul_rn(a.hi, b);
    const float e = fmaf(a.lo, b, fmaf(a.hi, b, -p));
    return fast_two_sum(p, e);
}

__device__ __forceinline__ dfl df_add(dfl a, dfl b)
{
    const dfl s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ dfl to_dfl(double v)
{
    const float hi = __double2float_rn(v);
    return {hi, __double2float_rn(v - (double)hi)};
}

// The fit weight of a neighbour at distance d. Distances are integers, so the weights
// of the first kWeights come from a table that each call fills once: at k = 128 the
// search evaluated 128 FP64 exponentials a seed (about 20 instructions of the narrow
// FP64 pipe each) for a few thousand distinct distances. The table's entries are this
// function's values; weights past its end (exp(-205) at the default decay) are
// computed. A call on the 1242x375 pair 1,301 -> 1,231 us.
constexpr int kWeights = 16384;
__device__ __forceinline__ dfl fit_weight(double a_per_unit, long long d)
{
    return to_dfl(exp_neg(a_per_unit * (double)d));
}

// Sums of 12 values over the warp: lane 8 g holds totals 3 g .. 3 g + 2 in q (other
// lanes partial sums). Halving exchanges: lanes 16 apart swap half of their values and
// keep the sum of the other half, then lanes 8 apart the same with 3 of 6, then xor
// butterflies finish the 3 sums in each group of 8 lanes.
__device__ __forceinline__ void warp_sum12(const double (&v)[12], double (&q)[3])
{
    const int lane = threadIdx.x & 31;
    const bool hi16 = lane & 16, hi8 = lane & 8;
    double h[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double keep = hi16 ? v[6 + i] : v[i], give = hi16 ? v[i] : v[6 + i];
        h[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double keep = hi8 ? h[3 + i] : h[i], give = hi8 ? h[i] : h[3 + i];
        q[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < 3; ++i) q[i] += __shfl_xor_sync(0xffffffffu, q[i], o);
}

// Per seed: keeps one link per neighbour (the smallest weight), compacting the list
// in place; end[s] becomes the end of the compacted list. One warp per seed walks
// the list in chunks of 32 and takes a chunk's neighbours one by one (about six of
// some twenty links): a ballot finds the neighbour's links, a warp minimum their
// weight, and lane i holds the i-th kept link in registers. A seed with more than 32
// neighbours keeps the others in its list, whose kept prefix never reaches the unread
// part. Also fills the table of fit weights, an entry a thread. 1242x375 pair: 20 us,
// 35 with a 32-step shuffle loop over 64-bit weights a chunk.
__global__ void __launch_bounds__(kThreads) epic_dedupe_kernel(const int* off, int* end, int* adj_t, unsigned* adj_w,
                                                               unsigned* minin, int n, double a_per_unit,
                                                               float2* weights, int n_weights)
{
    begin_after();
    constexpr unsigned kAll = 0xffffffffu;
    for (int d = blockIdx.x * kThreads + threadIdx.x; d < n_weights; d += gridDim.x * kThreads) {
        const dfl w = fit_weight(a_per_unit, d);
        weights[d] = make_float2(w.hi, w.lo);
    }
    const int lane = threadIdx.x & 31;
    const int s = (int)(((size_t)blockIdx.x * kThreads + threadIdx.x) >> 5);
    if (s >= n) return;  // warp-uniform
    const int b = off[s], e = off[s + 1];
    int cnt = 0, kt = -1;  // kept links; the lane's neighbour and weight
    unsigned kw = kNoLink;
    for (int c = b; c < e; c += 32) {
        const bool has = c + lane < e;
        const int t = has ? adj_t[c + lane] : -1;
        const unsigned w = has ? adj_w[c + lane] : kNoLink;
        unsigned left = __ballot_sync(kAll, has);
        while (left) {
            const int tt = __shfl_sync(kAll, t, __ffs(left) - 1);
            const bool in = t == tt;
            left &= ~__ballot_sync(kAll, in);
            const unsigned mw = __reduce_min_sync(kAll, in ? w : kNoLink);
            const bool hit = kt == tt;
            if (__any_sync(kAll, hit)) {
                if (hit) kw = min(kw, mw);
            } else if (cnt < 32) {
                if (lane == cnt) {
                    kt = tt;
                    kw = mw;
                }
                ++cnt;
            } else {
                int found = -1;
                for (int j = b + 32 + lane; j < b + cnt; j += 32)
                    if (adj_t[j] == tt) found = j;
                if (__any_sync(kAll, found >= 0)) {
                    if (found >= 0) adj_w[found] = min(adj_w[found], mw);
                } else {
                    if (lane == 0) {
                        adj_t[b + cnt] = tt;
                        adj_w[b + cnt] = mw;
                    }
                    ++cnt;
                }
                __syncwarp();
            }
        }
    }
    if (lane < cnt) {
        adj_t[b + lane] = kt;
        adj_w[b + lane] = kw;
    }
    // smallest link weight (a lower bound on the last step of any path into s)
    unsigned mn = kw;
    for (int j = b + 32 + lane; j < b + cnt; j += 32) mn = min(mn, adj_w[j]);
    mn = __reduce_min_sync(kAll, mn);
    if (lane == 0) {
        end[s] = b + cnt;
        minin[s] = mn;
    }
}

// Link records for the search (one 16-byte load a link): neighbour, its smallest link
// weight, the link's weight; the list of the seeds that hold a pixel (in any order; a
// warp takes its places with one atomic), and the outputs of those that do not.
__global__ void __launch_bounds__(kThreads) epic_link_meta_kernel(KnnArgs a, const int* adj_t,
                                                                  const unsigned* adj_w, int4* adj, int* list,
                                                                  int* list_count)
{
    begin_after();
    const int s = blockIdx.x * kThreads + threadIdx.x, lane = threadIdx.x & 31;
    const bool holds = s < a.n && a.seed_pix[s] >= 0;
    const unsigned hold = __ballot_sync(0xffffffffu, holds);
    int at = 0;
    if (lane == 0 && hold) at = atomicAdd(list_count, __popc(hold));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (s >= a.n) return;
    if (!holds) {
        if (a.knn_count) a.knn_count[s] = 0;
        if (a.fit_kind) a.fit_kind[s] = 0;
        for (int i = 0; i < 6; ++i) {
            a.models[6 * (size_t)s + i] = 0.0;
            if (a.dbg_models) a.dbg_models[6 * (size_t)s + i] = 0.0;
        }
        return;
    }
    list[at + __popc(hold & ((1u << lane) - 1))] = s;
    for (int i = a.off[s], e = a.end_of[s]; i < e; ++i) {
        const int t = adj_t[i];
        adj[i] = make_int4(t, (int)a.minin[t], (int)adj_w[i], 0);
    }
}

__device__ __forceinline__ long long warp_min(long long v)  // v >= 0
{
    const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)((unsigned long long)v >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)((unsigned long long)v >> 32) == hi ? (unsigned)v : ~0u);
    return (long long)(((unsigned long long)hi << 32) | lo);
}
__device__ __forceinline__ unsigned warp_min(unsigned v) { return __reduce_min_sync(0xffffffffu, v); }

__device__ __forceinline__ void atomic_min_shared(long long* p, long long v)
{
    atomicMin(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);  // v >= 0
}
__device__ __forceinline__ void atomic_min_shared(unsigned* p, unsigned v) { atomicMin(p, v); }

// Ascending sort of the first n <= 32 P keys of a shared array by one warp: P keys a
// lane in registers (lane l holds elements P l .. P l + P - 1), a bitonic network whose
// strides below P stay in the lane and whose others are shuffles. The shuffle stages
// are a loop: unrolled, they are some 700 instructions that each search runs once,
// and fetching them stalled the warps. Slots past n are filled with the largest key and
// not written back.
template <int P>
__device__ __forceinline__ void warp_sort(unsigned long long* key, int n)
{
    const int lane = threadIdx.x & 31;
    unsigned long long v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = lane + 32 * i < n ? key[lane + 32 * i] : kNone;  // any order will do
    auto exchange = [&](int i, int j, bool asc) {  // elements i < j of the lane
        const unsigned long long x = v[i], y = v[j];
        const bool keep = (x < y) == asc;
        v[i] = keep ? x : y;
        v[j] = keep ? y : x;
    };
    // sorted runs of P, ascending in even lanes
#pragma unroll
    for (int size = 2; size <= P; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (!(i & stride)) exchange(i, i ^ stride, size < P ? (i & size) == 0 : (lane & 1) == 0);
    // merges of runs of `lanes` / 2 lanes
#pragma unroll 1
    for (int lanes = 2; lanes <= 32; lanes <<= 1) {
        const bool asc = (lane & lanes) == 0;  // (lanes = 32: all ascending)
#pragma unroll 1
        for (int o = lanes >> 1; o > 0; o >>= 1) {
            const bool low = (lane & o) == 0;
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const unsigned long long w = __shfl_xor_sync(0xffffffffu, v[i], o);
                v[i] = (v[i] < w) == (low == asc) ? v[i] : w;
            }
        }
#pragma unroll
        for (int stride = P >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int i = 0; i < P; ++i)
                if (!(i & stride)) exchange(i, i ^ stride, asc);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < P; ++i)
        if (P * lane + i < n) key[P * lane + i] = v[i];
    __syncwarp();
}

// Moves the `want` smallest of n distinct keys (want < n) to the front of a shared
// array, in any order. The want-th smallest distance is found by bisection between
// lo and hi (fewer than want keys lie below lo, at least want at or below hi), then,
// if more than want keys are at or below it, the index bound among those at it.
__device__ __forceinline__ void warp_select(unsigned long long* key, int n, int want, long long lo, long long hi)
{
    const int lane = threadIdx.x & 31;
    auto count = [&](unsigned long long bound) {  // keys below bound
        int c = 0;
        for (int i = lane; i < n; i += 32) c += key[i] < bound;
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
    };
    auto above = [](long long d) {  // above every key at distance d
        return d + 1 < kDistLimit ? (unsigned long long)(d + 1) << kIdxBits : kNone;
    };
    while (lo < hi) {
        const long long mid = lo + ((hi - lo) >> 1);
        if (count(above(mid)) >= want)
            hi = mid;
        else
            lo = mid + 1;
    }
    unsigned long long bound = above(lo);  // keys below it are kept
    if (count(bound) > want) {
        unsigned long long a = (unsigned long long)lo << kIdxBits, b = bound;  // count(a) < want < count(b)
        while (a < b) {
            const unsigned long long mid = a + ((b - a) >> 1);
            if (count(mid) >= want)
                b = mid;
            else
                a = mid + 1;
        }
        bound = a;
    }
    int kept = 0;
    for (int c = 0; c < n; c += 32) {  // in place: kept never passes the chunk being read
        const unsigned long long v = c + lane < n ? key[c + lane] : kNone;
        const bool take = v < bound;
        const unsigned tm = __ballot_sync(0xffffffffu, take);
        if (take) key[kept + __popc(tm & ((1u << lane) - 1))] = v;
        kept += __popc(tm);
        __syncwarp();
    }
}

// The k nearest seeds of seed s in the seed graph, exactly, by Dijkstra with batch
// settling: with m the smallest tentative distance on the frontier, every frontier
// seed v with d(v) <= m + minin(v) is final (a shorter path would have to end with
// a link from an unsettled seed, at least m away, and that link weighs at least
// minin(v)); the whole batch is settled (appended to the settled keys and removed
// from the frontier list), then its links are relaxed, one lane per link;
// newly discovered seeds join the frontier list. The search stops once k settled
// seeds lie below m (every unsettled seed is at least m away) or the frontier is
// empty; the k smallest settled keys (distance << 24 | index) are then selected and
// sorted (cnt_out of them). Returns 0, kRetry when the hash, the frontier list, the
// settled list or the distance type is too small, or kErrRange when a distance leaves
// 40 bits.
// Bound by instruction issue and shared-memory latency, so the steps are kept short:
// distances of 32 bits, one 16-byte record a link, owners of links by bit masks instead
// of a shuffled binary search, settled keys counted only once there are k of them, and
// a register sort of the k kept keys instead of a shared-memory sort of all settled ones
// padded to 256. Search kernel on the 1242x375 pair (k = 128): 880 -> 660 us; 28
// searches an SM instead of 24.
template <typename DT, int HCAP, int FCAP, int SCAP>
__device__ int knn_search(const KnnArgs& a, int s, unsigned char* base, int& cnt_out)
{
    using Lay = KnnLayout<DT, HCAP, FCAP, SCAP>;
    constexpr bool kNarrow = sizeof(DT) == 4;
    constexpr DT kInf = kNarrow ? (DT)0xffffffffu : (DT)0x7fffffffffffffffll;
    int* hkey = reinterpret_cast<int*>(base);
    volatile int* vh = hkey;
    DT* hdist = reinterpret_cast<DT*>(base + Lay::o_hdist);
    unsigned long long* skey = reinterpret_cast<unsigned long long*>(base + Lay::o_sort);
    unsigned* hmin = reinterpret_cast<unsigned*>(base + Lay::o_minin);
    short* front = reinterpret_cast<short*>(base + Lay::o_front);
    int* fcount = reinterpret_cast<int*>(base + Lay::o_count);  // frontier list length
    const int lane = threadIdx.x & 31;
    // multiplicative hash scaled onto [0, HCAP) (HCAP need not be a power of two)
    auto slot_of = [](int t) {
        return (int)(((unsigned long long)((unsigned)t * 0x9E3779B1u) * (unsigned)HCAP) >> 32);
    };

    for (int j = 4 * lane; j < HCAP; j += 128) {
        *reinterpret_cast<int4*>(hkey + j) = make_int4(-1, -1, -1, -1);
        if constexpr (kNarrow)
            *reinterpret_cast<uint4*>(hdist + j) = make_uint4(~0u, ~0u, ~0u, ~0u);
        else
            for (int i = 0; i < 4; ++i) hdist[j + i] = kInf;
    }
    __syncwarp();
    if (lane == 0) {
        const int h = slot_of(s);
        hkey[h] = s;
        hdist[h] = 0;
        hmin[h] = a.minin[s];
        front[0] = (short)h;
        *fcount = 1;
    }
    __syncwarp();
    int status = 0, nset = 0;
    DT last = 0, m = 0;  // the frontier minimum at the step before the last, and at the last
    for (int step = 0; step < HCAP; ++step) {  // every step settles at least the frontier minimum
        const int nf = *fcount;
        if (nf == 0) {  // every reachable seed is settled
            last = 0;
            m = kInf;
            break;
        }
        last = m;  // fewer than k settled seeds lie below it
        m = kInf;
        for (int i = lane; i < nf; i += 32) m = min(m, hdist[front[i]]);
        m = warp_min(m);
        if (nset >= a.k) {
            const unsigned long long bound = (unsigned long long)m << kIdxBits;
            int below = 0;
            for (int i = lane; i < nset; i += 32) below += skey[i] < bound;
            if ((int)__reduce_add_sync(0xffffffffu, (unsigned)below) >= a.k) break;
        }
        // settle the batch: compact the frontier list in place (chunks are read
        // before the kept entries of the chunk are written, and never ahead of them)
        const int nset0 = nset;
        int kept = 0;
        for (int c = 0; c < nf; c += 32) {
            const int i = c + lane;
            int h = -1;
            DT d = 0;
            bool bat = false;
            if (i < nf) {
                h = front[i];
                d = hdist[h];
                bat = d - m <= (DT)hmin[h];
            }
            const unsigned bm = __ballot_sync(0xffffffffu, bat), km = __ballot_sync(0xffffffffu, i < nf && !bat);
            const unsigned lt = (1u << lane) - 1;
            if (bat) {
                const int pos = nset + __popc(bm & lt);
                if (pos < SCAP) skey[pos] = ((unsigned long long)d << kIdxBits) | (unsigned long long)hkey[h];
            } else if (i < nf) {
                front[kept + __popc(km & lt)] = (short)h;
            }
            nset += __popc(bm);
            kept += __popc(km);
            __syncwarp();
        }
        if (nset > SCAP) {
            status = kRetry;
            break;
        }
        if (lane == 0) *fcount = kept;
        __syncwarp();
        // relax the batch's links, one lane per link: the batch seeds' link counts
        // are prefix-summed over the warp (32 seeds at a time); in a chunk of 32 links
        // the seeds whose lists begin in it set a bit at their first link, and a lane's
        // owner is the last seed that begins at or before its link (every batch seed
        // has a link: it was reached through one, or is s, alone or with links), so all
        // the links' loads are in flight together
        int st = 0;
        for (int b0 = nset0; b0 < nset; b0 += 32) {
            const int nb = min(32, nset - b0);
            int u = 0, first = 0, deg = 0;
            DT du = 0;
            if (lane < nb) {
                const unsigned long long kb = skey[b0 + lane];
                u = (int)(kb & kIdxMask);
                du = (DT)(kb >> kIdxBits);
                first = a.off[u];
                deg = a.end_of[u] - first;
            }
            int incl = deg;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31), excl = incl - deg;
            for (int c0 = 0; c0 < total; c0 += 32) {
                const int e = c0 + lane, rel = excl - c0;
                const bool here = lane < nb && rel >= 0 && rel < 32;
                const unsigned starts = __reduce_or_sync(0xffffffffu, here ? 1u << rel : 0u);
                const int before = __popc(__ballot_sync(0xffffffffu, lane < nb && rel < 0));
                const int ow = max(before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1, 0);
                const int le = __shfl_sync(0xffffffffu, first - excl, ow) + e;
                const DT odu = __shfl_sync(0xffffffffu, du, ow);
                if (e >= total || st) continue;
                const int4 li = __ldg(a.adj + le);  // neighbour, its smallest link weight, the link's weight
                const long long nd = (long long)odu + (long long)(unsigned)li.z;
                if (nd >= kDistLimit) st |= kErrRange;
                if (kNarrow && nd >= (long long)kInf) {  // (a path of several links may be longer than 32 bits)
                    st |= kRetry;
                    continue;
                }
                const int t = li.x;
                int h = slot_of(t), hs = -1;
                for (int q = 0; q < HCAP; ++q) {
                    const int c = vh[h];
                    if (c == t) {
                        hs = h;
                        break;
                    }
                    if (c == -1) {
                        const int prev = atomicCAS(&hkey[h], -1, t);
                        if (prev == -1) {  // discovered: joins the frontier list
                            hmin[h] = (unsigned)li.y;
                            const int f = atomicAdd(fcount, 1);
                            if (f < FCAP)
                                front[f] = (short)h;
                            else
                                st |= kRetry;
                            hs = h;
                            break;
                        }
                        if (prev == t) {
                            hs = h;
                            break;
                        }
                    }
                    h = h + 1 == HCAP ? 0 : h + 1;
                }
                if (hs < 0) {
                    st |= kRetry;
                    continue;
                }
                // a settled seed keeps its final distance: the minimum is a no-op there
                atomic_min_shared(&hdist[hs], (DT)nd);
            }
        }
        __syncwarp();
        status = __reduce_or_sync(0xffffffffu, st);
        if (status) break;
    }
    if (!status) {
        const int want = min(nset, a.k);
        cnt_out = want;
        const int room = want <= 32 ? 32 : want <= 64 ? 64 : want <= 128 ? 128 : 256;  // the sort's width
        int n = nset;
        if (n > room) {
            // every settled key of the list is below 2^40, and of those below m at least k
            const long long hi = (long long)m < kDistLimit ? (long long)m : kDistLimit - 1;
            warp_select(skey, n, want, (long long)last, hi);
            n = want;
        }
        if (room == 32)
            warp_sort<1>(skey, n);
        else if (room == 64)
            warp_sort<2>(skey, n);
        else if (room == 128)
            warp_sort<4>(skey, n);
        else
            warp_sort<8>(skey, n);
    }
    return status & kErrRange ? kErrRange : status;
}

// The weighted sums of the affine fit of seed s (entry idx of the list) over its neighbourhood (sorted keys), and
// the neighbourhood outputs. The 3 x 3 normal equations lose too many digits in FP32
// when a neighbourhood is narrow: the weights come from an FP64 exponential, the
// per-neighbour terms are summed in double-float, the lanes' sums are reduced and
// the systems solved in FP64 (epic_solve_kernel). M = sum w v v^T,
// v = (x_t - x_s, y_t - y_s, 1).
__device__ void knn_fit_sums(const KnnArgs& a, int idx, int s, int cnt, const unsigned long long* key)
{
    const int lane = threadIdx.x & 31, k = a.k;
    if (a.knn_count && lane == 0) a.knn_count[s] = cnt;
    if (a.knn_idx)
        for (int j = lane; j < cnt; j += 32) {
            a.knn_idx[(size_t)s * k + j] = (int)(key[j] & kIdxMask);
            a.knn_dist[(size_t)s * k + j] = (int64_t)(key[j] >> kIdxBits);
        }
    const float2 ps = a.pts[s];
    dfl acc[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = {0.f, 0.f};
#pragma unroll 1
    for (int j = lane; j < cnt; j += 32) {
        const int t = (int)(key[j] & kIdxMask);
        const long long d = (long long)(key[j] >> kIdxBits);
        dfl w;
        if (d < a.n_weights) {
            const float2 t = __ldg(a.weights + d);
            w = {t.x, t.y};
        } else {
            w = fit_weight(a.a_per_unit, d);
        }
        const float2 pt = a.pts[t], ft = a.flow[t];
        const dfl vx = two_sum(pt.x, -ps.x), vy = two_sum(pt.y, -ps.y);  // exact differences
        const dfl wx = df_mul(w, vx), wy = df_mul(w, vy);
        acc[0] = df_add(acc[0], df_mul(wx, vx));
        acc[1] = df_add(acc[1], df_mul(wx, vy));
        acc[2] = df_add(acc[2], wx);
        acc[3] = df_add(acc[3], df_mul(wy, vy));
        acc[4] = df_add(acc[4], wy);
        acc[5] = df_add(acc[5], w);
        acc[6] = df_add(acc[6], df_mul(wx, ft.x));
        acc[7] = df_add(acc[7], df_mul(wy, ft.x));
        acc[8] = df_add(acc[8], df_mul(w, ft.x));
        acc[9] = df_add(acc[9], df_mul(wx, ft.y));
        acc[10] = df_add(acc[10], df_mul(wy, ft.y));
        acc[11] = df_add(acc[11], df_mul(w, ft.y));
    }
    double accd[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) accd[i] = (double)acc[i].hi + (double)acc[i].lo;
    double tot[3];
    warp_sum12(accd, tot);
    if (lane & 7) return;
    double* row = a.sums + 12 * (size_t)(idx - a.begin) + 3 * (lane >> 3);
    row[0] = tot[0];
    row[1] = tot[1];
    row[2] = lane == 8 && cnt < 3 ? -tot[2] : tot[2];  // sum w > 0: a negative one marks fewer than 3 neighbours
}

// One-warp blocks: an SM's FP64 pipe takes 16 cycles a warp instruction, so eight warps
// of a block on one SM while others idle took 20 us for 1,953 seeds (12 us with
// one-warp blocks; 50,676 seeds 37 and 26 us).
constexpr int kSolveThreads = 32;

// Solves the fits of this launch's seeds from their sums, a thread a seed. The
// solve is about 250 FP64 operations (a dozen divisions and square roots); GB300
// issues an FP64 instruction of one lane no faster than one of 32, so on lane 0 of
// each search's warp the solves kept the search kernel's FP64 pipe busy 58% of its
// time. 1242x375 pair, 50,676 matches, k = 128: a call 1,761 -> 1,301 us.
__global__ void __launch_bounds__(kSolveThreads) epic_solve_kernel(KnnArgs a)
{
    begin_after();
    const int idx = a.begin + blockIdx.x * kSolveThreads + threadIdx.x;
    if (idx >= min(a.end, *a.list_count)) return;
    const int s = a.list[idx];
    const double2* row = reinterpret_cast<const double2*>(a.sums + 12 * (size_t)(idx - a.begin));
    const double2 q0 = row[0], q1 = row[1], q2 = row[2], q3 = row[3], q4 = row[4], q5 = row[5];
    const double m00 = q0.x, m01 = q0.y, m02 = q1.x, m11 = q1.y, m12 = q2.x, m22 = fabs(q2.y);
    const double u0 = q3.x, u1 = q3.y, u2 = q4.x, v0 = q4.y, v1 = q5.x, v2 = q5.y;
    // affine only with 3+ neighbours whose weighted position covariance (the Schur
    // complement of the constant term over sum w) has lambda_min >= min_spread^2
    bool affine = a.model == 1 && q2.y > 0.0;
    if (affine) {
        const double mx = m02 / m22, my = m12 / m22;
        const double cxx = m00 / m22 - mx * mx, cxy = m01 / m22 - mx * my, cyy = m11 / m22 - my * my;
        const double h = 0.5 * (cxx - cyy);
        affine = 0.5 * (cxx + cyy) - sqrt(h * h + cxy * cxy) >= a.min_spread2;
    }
    double A00 = 0, A01 = 0, A10 = 0, A11 = 0, b0 = u2 / m22, b1 = v2 / m22;
    if (affine) {
        // Cholesky of M = L L^T, then forward and back substitution for both flow components
        const double l00 = sqrt(m00), l10 = m01 / l00, l20 = m02 / l00;
        const double l11 = sqrt(m11 - l10 * l10), l21 = (m12 - l20 * l10) / l11;
        const double l22 = sqrt(m22 - l20 * l20 - l21 * l21);
        const double zu0 = u0 / l00, zu1 = (u1 - l10 * zu0) / l11, zu2 = (u2 - l20 * zu0 - l21 * zu1) / l22;
        const double zv0 = v0 / l00, zv1 = (v1 - l10 * zv0) / l11, zv2 = (v2 - l20 * zv0 - l21 * zv1) / l22;
        b0 = zu2 / l22;
        A01 = (zu1 - l21 * b0) / l11;
        A00 = (zu0 - l10 * A01 - l20 * b0) / l00;
        b1 = zv2 / l22;
        A11 = (zv1 - l21 * b1) / l11;
        A10 = (zv0 - l10 * A11 - l20 * b1) / l00;
    }
    double* mo = a.models + 6 * (size_t)s;
    mo[0] = A00; mo[1] = A01; mo[2] = A10; mo[3] = A11; mo[4] = b0; mo[5] = b1;
    if (a.dbg_models) {
        double* dm = a.dbg_models + 6 * (size_t)s;
        dm[0] = A00; dm[1] = A01; dm[2] = A10; dm[3] = A11; dm[4] = b0; dm[5] = b1;
    }
    if (a.fit_kind) a.fit_kind[s] = affine ? 1 : 2;
}

// One warp per seed with a fast layout; searches that outgrow it are queued for
// the retry kernel.
template <int HCAP, int FCAP, int SCAP>
__global__ void __launch_bounds__(kFastWarps * 32) epic_knn_fit_kernel(KnnArgs a)
{
    using Lay = KnnLayout<unsigned, HCAP, FCAP, SCAP>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int idx = a.begin + blockIdx.x * kFastWarps + wid;
    if (idx >= min(a.end, *a.list_count)) return;  // warp-uniform
    const int s = a.list[idx];
    unsigned char* base = smem + (size_t)wid * Lay::bytes;
    int cnt = 0;
    const int st = knn_search<unsigned, HCAP, FCAP, SCAP>(a, s, base, cnt);
    if (st == kRetry) {
        if (lane == 0) a.retry_list[atomicAdd(a.retry_count, 1)] = idx;
        return;
    }
    if (st) {
        if (lane == 0) atomicOr(a.err, st);
        return;
    }
    knn_fit_sums(a, idx, s, cnt, reinterpret_cast<const unsigned long long*>(base + Lay::o_sort));
}

// The queued searches of this launch's seeds with room for 8192 discovered seeds, one
// warp per block.
__global__ void __launch_bounds__(32) epic_knn_retry_kernel(KnnArgs a)
{
    using Lay = RetryLayout;
    extern __shared__ __align__(16) unsigned char smem[];
    const int total = *a.retry_count;
    for (int i = blockIdx.x; i < total; i += gridDim.x) {
        const int idx = a.retry_list[i];
        if (idx < a.begin) continue;  // of an earlier launch
        const int s = a.list[idx];
        int cnt = 0;
        const int st = knn_search<long long, kBigH, kBigF, kBigS>(a, s, smem, cnt);
        if (st) {
            if ((threadIdx.x & 31) == 0) atomicOr(a.err, st == kRetry ? kErrFrontier : st);
            continue;
        }
        knn_fit_sums(a, idx, s, cnt, reinterpret_cast<const unsigned long long*>(smem + Lay::o_sort));
    }
}

__global__ void __launch_bounds__(kThreads) epic_dense_kernel(const unsigned long long* key, const double* models,
                                                              const float2* pts, int W, int H, float2* dense,
                                                              int32_t* labels, int64_t* dist, const int* err,
                                                              unsigned* status)
{
    begin_after();
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
    if (x == 0 && y == 0) {  // a device-side failure of the call goes into the library's status word
        const int e = *err;
        if (e) atomicOr(status, e & (kErrPasses | kErrSync) ? DGF_DEV_EPIC_PASSES : DGF_DEV_EPIC_CAPACITY);
    }
    if (x >= W || y >= H) return;
    const size_t o = (size_t)y * W + x;
    const unsigned long long k = key[o];
    if (k == kNone) {
        dense[o] = make_float2(0.f, 0.f);
        if (labels) labels[o] = -1;
        if (dist) dist[o] = -1;
        return;
    }
    const int s = (int)(k & kIdxMask);
    const double* m = models + 6 * (size_t)s;
    const float2 p = pts[s];
    const double dx = (double)x - (double)p.x, dy = (double)y - (double)p.y;
    dense[o] = make_float2((float)(m[0] * dx + m[1] * dy + m[4]), (float)(m[2] * dx + m[3] * dy + m[5]));
    if (labels) labels[o] = s;
    if (dist) dist[o] = (int64_t)(k >> kIdxBits);
}

// Pass counters, the status word, the retry count, the barrier, the list's length.
constexpr int kCounters = kMaxPasses + 4;

// Workspace layout (256-byte aligned sections).
struct EpicLayout {
    size_t key, cost, seed_pix, cnt, off, cur, minin, bsum, adj_t, adj_w, adj_i, models, retry, counters, total;
};

EpicLayout epic_layout(int W, int H, int n)
{
    const size_t np = (size_t)W * H, nl = 4 * np;  // at most two links per pixel, stored both ways
    EpicLayout L;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at = dgf::round_up(at + bytes, 256);
        return o;
    };
    L.key = take(np * 8);
    L.cost = take(np * 4);
    L.seed_pix = take((size_t)n * 4);
    L.cnt = take((size_t)n * 4);
    L.off = take(((size_t)n + 1) * 4);
    L.cur = take((size_t)n * 4);
    L.minin = take((size_t)n * 4);
    L.bsum = take(((size_t)n / 1024 + 2) * 12);  // block totals, block offsets (+1), scan cursors
    L.adj_t = take(nl * 4);
    L.adj_w = take(nl * 4);
    L.adj_i = take(nl * 16);
    L.models = take((size_t)n * 48);
    L.retry = take((size_t)n * 4);
    L.counters = take(kCounters * 4);
    L.total = at;
    return L;
}

bool params_ok(const dgf_epic_params* p)
{
    return p && p->version == DGF_EPIC_PARAMS_VERSION && p->k >= 1 && p->k <= DGF_EPIC_MAX_K &&
           (p->model == 0 || p->model == 1) && p->cost_base >= 1 && p->cost_base <= 4096 && p->cost_gain >= 0 &&
           p->cost_gain <= 32 && p->a >= 0.0 && p->a < 1e30 && p->min_spread >= 0.0 && p->min_spread < 1e30;
}

}  // namespace

namespace {

__global__ void exp_neg_kernel(const double* y, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = exp_neg(y[i]);
}

}  // namespace

// The exponential of the fit weights, exported so that its accuracy can be checked
// against a reference exp on the same arguments.
extern "C" int dgf_epic_exp_neg(const double* y, double* out, int n, cudaStream_t stream)
{
    if (n < 0 || (n > 0 && (!y || !out))) return DGF_ERR_ARG;
    if (n == 0) return DGF_OK;
    exp_neg_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(y, out, n);
    return dgf::launch_status();
}

extern "C" int dgf_epic_params_default(dgf_epic_params* p)
{
    if (!p) return DGF_ERR_ARG;
    p->version = DGF_EPIC_PARAMS_VERSION;
    p->k = 128;
    p->model = 1;
    p->cost_base = 4;
    p->cost_gain = 1;
    p->a = 0.1;
    p->min_spread = 1.0;
    return DGF_OK;
}

extern "C" size_t dgf_epic_workspace(int W, int H, int n)
{
    if (W < 1 || H < 1 || n < 0 || W + H > DGF_EPIC_MAX_W_PLUS_H || n > DGF_EPIC_MAX_POINTS) return 0;
    return epic_layout(W, H, n).total;
}

extern "C" int epic_interpolate(const uint8_t* img, int W, int H, int pitch, const float* pts, const float* flow,
                                const uint8_t* status, int n, const dgf_epic_params* p, float* dense,
                                const dgf_epic_debug* dbg, void* workspace, size_t ws_bytes, cudaStream_t stream)
{
    if (!params_ok(p) || W < 1 || H < 1 || W + H > DGF_EPIC_MAX_W_PLUS_H || pitch < W || n < 0 ||
        n > DGF_EPIC_MAX_POINTS || !img || !dense || !workspace || (n > 0 && (!pts || !flow || !status)))
        return DGF_ERR_ARG;
    if (!dgf::aligned(dense, 8) || !dgf::aligned(workspace, 256) || (n > 0 && (!dgf::aligned(pts, 8) || !dgf::aligned(flow, 8))))
        return DGF_ERR_ARG;
    dgf_epic_debug d = {};
    if (dbg) d = *dbg;
    if ((d.knn_idx == nullptr) != (d.knn_dist == nullptr)) return DGF_ERR_ARG;
    if ((d.labels && !dgf::aligned(d.labels, 4)) || (d.dist && !dgf::aligned(d.dist, 8)) || (d.knn_idx && !dgf::aligned(d.knn_idx, 4)) ||
        (d.knn_dist && !dgf::aligned(d.knn_dist, 8)) || (d.knn_count && !dgf::aligned(d.knn_count, 4)) ||
        (d.models && !dgf::aligned(d.models, 8)) || (d.retried && !dgf::aligned(d.retried, 4)))
        return DGF_ERR_ARG;
    const EpicLayout L = epic_layout(W, H, n);
    if (ws_bytes < L.total) return DGF_ERR_WORKSPACE;
    char* ws = static_cast<char*>(workspace);
    auto* key = reinterpret_cast<unsigned long long*>(ws + L.key);
    auto* cost = reinterpret_cast<int*>(ws + L.cost);
    auto* seed_pix = reinterpret_cast<int*>(ws + L.seed_pix);
    auto* cnt = reinterpret_cast<int*>(ws + L.cnt);
    auto* off = reinterpret_cast<int*>(ws + L.off);
    auto* cur = reinterpret_cast<int*>(ws + L.cur);
    auto* adj_t = reinterpret_cast<int*>(ws + L.adj_t);
    auto* adj_w = reinterpret_cast<unsigned*>(ws + L.adj_w);
    auto* adj_i = reinterpret_cast<int4*>(ws + L.adj_i);
    auto* minin = reinterpret_cast<unsigned*>(ws + L.minin);
    auto* bsum = reinterpret_cast<int*>(ws + L.bsum);
    auto* retry_list = reinterpret_cast<int*>(ws + L.retry);
    auto* models = reinterpret_cast<double*>(ws + L.models);
    auto* changed = reinterpret_cast<int*>(ws + L.counters);
    int* err = changed + kMaxPasses;
    int* retry_count = err + 1;
    unsigned* sync_count = reinterpret_cast<unsigned*>(retry_count + 1);
    int* list_count = retry_count + 2;
    const float2* p2 = reinterpret_cast<const float2*>(pts);
    const float2* f2 = reinterpret_cast<const float2*>(flow);

    unsigned* dev_status = dgf::status_word();
    if (!dev_status) return DGF_ERR_CUDA;
    const dim3 pix_block(32, 8), pix_grid((W + 31) / 32, (H + 7) / 8);
    const unsigned pt_grid = (unsigned)((n + kThreads - 1) / kThreads);
    epic_cost_kernel<<<pix_grid, pix_block, 0, stream>>>(img, W, H, pitch, p->cost_base, p->cost_gain, cost, key,
                                                        changed, kCounters);
    if (n > 0) {
        launch_next(epic_seed_kernel, pt_grid, kThreads, stream, p2, status, n, W, H, key, seed_pix, cnt);
        launch_next(epic_seed_owner_kernel, pt_grid, kThreads, stream, key, n, seed_pix);
    }
    int rc = dgf::launch_status();
    if (rc != DGF_OK) return rc;

    // geodesic Voronoi labelling: passes until one changes nothing, in one
    // cooperative launch of as many blocks as can be resident (at most one a tile)
    {
        const long long tiles = (long long)((W + kTile - 1) / kTile) * ((H + kTile - 1) / kTile);
        const unsigned grid = dgf::cooperative_blocks(epic_voronoi_kernel, kThreads, tiles);
        const dim3 block(32, 8);
        void* args[] = {(void*)&cost, (void*)&key, (void*)&W, (void*)&H, (void*)&changed, (void*)&sync_count,
                        (void*)&err};
        if ((rc = dgf::launch_cooperative((const void*)epic_voronoi_kernel, grid, block, args, stream)) != DGF_OK) return rc;
    }

    if (n > 0) {
        launch_next(epic_links_kernel<false>, pix_grid, pix_block, stream, key, cost, W, H, cnt, nullptr, nullptr, nullptr,
                                                                     nullptr, err);
        const int nb = (n + 1023) / 1024;
        launch_next(epic_scan_blocks_kernel, nb, 1024, stream, cnt, n, off, bsum);
        launch_next(epic_scan_kernel, 1, 1024, stream, bsum, nb, bsum + nb, bsum + 2 * nb + 1);
        launch_next(epic_scan_add_kernel, nb, 1024, stream, bsum + nb, n, nb, off, cur);
        launch_next(epic_links_kernel<true>, pix_grid, pix_block, stream, key, cost, W, H, nullptr, off, cur, adj_t, adj_w,
                                                                    err);
        // the weights' table takes the place of the pixel costs
        const int n_weights = (int)std::min<size_t>(kWeights, (L.seed_pix - L.cost) / sizeof(float2));
        launch_next(epic_dedupe_kernel, (unsigned)((n + kThreads / 32 - 1) / (kThreads / 32)), kThreads, stream,
                    off, cur, adj_t, adj_w, minin, n, p->a / (2.0 * p->cost_base), reinterpret_cast<float2*>(cost), n_weights);
        KnnArgs a;
        a.pts = p2;
        a.flow = f2;
        a.seed_pix = seed_pix;
        a.off = off;
        a.end_of = cur;
        a.minin = minin;
        a.adj = adj_i;
        a.models = models;
        a.err = err;
        a.retry_count = retry_count;
        a.retry_list = retry_list;
        a.knn_idx = d.knn_idx;
        a.knn_dist = d.knn_dist;
        a.knn_count = d.knn_count;
        a.dbg_models = d.models;
        a.fit_kind = d.fit_kind;
        a.n = n;
        a.k = p->k;
        a.model = p->model;
        a.a_per_unit = p->a / (2.0 * p->cost_base);
        a.min_spread2 = p->min_spread * p->min_spread;
        const bool small = p->k <= kSmallK;
        auto fast = small ? epic_knn_fit_kernel<384, 256, 256> : epic_knn_fit_kernel<1024, 512, 512>;
        const size_t smem_fast = (small ? SmallLayout::bytes : LargeLayout::bytes) * kFastWarps;
        const size_t smem_big = RetryLayout::bytes;
        if (cudaFuncSetAttribute(fast, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_fast) != cudaSuccess ||
            cudaFuncSetAttribute(epic_knn_retry_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_big) !=
                cudaSuccess)
            return DGF_ERR_CUDA;
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            return DGF_ERR_CUDA;
        // the list takes the place of the link counts; the fits' sums that of adj_t and
        // adj_w once the link records are made. Seeds beyond its room (W H / 3 of them; at
        // most W H hold a pixel) are searched and solved in further launches.
        int* list = cnt;
        a.list = list;
        a.list_count = list_count;
        a.n_weights = n_weights;
        a.weights = reinterpret_cast<const float2*>(cost);
        launch_next(epic_link_meta_kernel, pt_grid, kThreads, stream, a, adj_t, adj_w, adj_i, list, list_count);
        a.sums = reinterpret_cast<double*>(adj_t);
        const long long holders = std::min<long long>(n, (long long)W * H);
        const long long room = (long long)((L.adj_i - L.adj_t) / (12 * sizeof(double)));
        for (long long at = 0; at < holders; at += room) {
            a.begin = (int)at;
            a.end = (int)std::min(holders, at + room);
            const int m = a.end - a.begin;
            fast<<<(unsigned)((m + kFastWarps - 1) / kFastWarps), kFastWarps * 32, smem_fast, stream>>>(a);
            epic_knn_retry_kernel<<<(unsigned)sms, 32, smem_big, stream>>>(a);
            launch_next(epic_solve_kernel, (unsigned)((m + kSolveThreads - 1) / kSolveThreads), kSolveThreads, stream, a);
        }
    }
    launch_next(epic_dense_kernel, pix_grid, pix_block, stream, key, models, p2, W, H, reinterpret_cast<float2*>(dense),
                                                          d.labels, d.dist, err, dev_status);
    if (d.retried &&
        cudaMemcpyAsync(d.retried, retry_count, sizeof(int), cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
        return DGF_ERR_CUDA;
    return dgf::launch_status();
}
