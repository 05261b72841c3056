// S2 - the depth sort of the visible Gaussians (Sec. 3.3: the Gaussians are
// sorted relative to the camera; the paper's renderer uses GPU radix sorts),
// and the scans of the prune entry points.
//
// The depth order is a stable LSD radix sort of the visible Gaussians, taken
// in index order, by the float bits of their depth (so ties keep index
// order).  It runs as
//   1. one pass over all Gaussians that counts the visible ones, the four
//      8-bit digit histograms of their keys and the smallest and largest key;
//   2. one kernel per digit.  A CTA takes a tile of 4096 items, ranks them
//      by digit in shared memory, and places every digit's run of the tile
//      at the count of that digit in all smaller keys (the histogram) plus
//      its count in the tiles before this one.  The first digit kernel reads
//      the Gaussians directly, keeps the visible ones and also writes their
//      indices in index order (the visible list of the backward).  Its tiles
//      are the histogram pass's, which counts the first digit per tile and
//      per group of G consecutive tiles (G^2 at or above the tile count): a
//      tile's prefix is the groups before its group plus the tiles before it
//      in its group: two threads per digit, one loading at most sqrt(tiles)
//      group counts and the other fewer than 2 sqrt(tiles) tile counts, all
//      independent loads.
//      The later digit kernels, over the visible Gaussians only, take their
//      tiles by ticket and find the prefix by a decoupled look-back over the
//      tiles before them (the single-pass prefix scan of Merrill and Garland,
//      used per digit as in Adinets and Merrill's Onesweep radix sort).
// A digit at and above the highest bit where the smallest and largest key
// differ is the same in every key: its kernel returns at once, and the last
// digit kernel that runs writes the final order.  A tile waits only on tiles
// with smaller tickets, whose CTAs are already running, and every wait is
// bounded (GS_ERR_TIMEOUT in the status word when it gives up).
//
// The scans of the prune entry points keep a fixed grid of sort_blocks() CTAs
// that each own a contiguous range of the items, so item counts produced on
// the device never need to travel to the host.
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ void block_range(uint32_t n, uint32_t &beg, uint32_t &end) {
    const uint64_t tiles = (static_cast<uint64_t>(n) + kSortTile - 1) / kSortTile;
    const uint64_t per = (tiles + gridDim.x - 1) / gridDim.x;
    const uint64_t b = static_cast<uint64_t>(blockIdx.x) * per * kSortTile;
    const uint64_t e = b + per * kSortTile;
    beg = static_cast<uint32_t>(b < n ? b : n);
    end = static_cast<uint32_t>(e < n ? e : n);
}

// Exclusive scan over the 256 threads of a block; *total = sum of all v.
__device__ __forceinline__ uint32_t block_scan_256(uint32_t v, uint32_t *s_w, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < 8 ? s_w[lane] : 0;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < 8) s_w[lane] = w;
    }
    __syncthreads();
    const uint32_t base = warp > 0 ? s_w[warp - 1] : 0;
    *total = s_w[7];
    __syncthreads();
    return base + x - v;
}

// ---------------------------------------------------------------------------
// Generic two-kernel scan: reduce per block, then rescan, each block first
// adding up the counts of the blocks before it (at most kMaxSortBlocks).

struct NSrc {               // item count: min(*dev, cap) if dev, else cap
    const uint32_t *dev;
    uint32_t cap;
    __device__ __forceinline__ uint32_t get() const {
        if (!dev) return cap;
        const uint32_t d = *dev;
        return d < cap ? d : cap;
    }
};

template <class F>
__global__ void __launch_bounds__(256) k_scan_reduce(F f, NSrc ns, uint32_t *__restrict__ partials) {
    chain_start();
    __shared__ uint32_t s_w[8];
    uint32_t beg, end;
    block_range(ns.get(), beg, end);
    uint32_t acc = 0;
    for (uint32_t i = beg + threadIdx.x; i < end; i += 256) acc += f(i);
    uint32_t tot;
    block_scan_256(acc, s_w, &tot);
    if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

template <class F, class Out>
__global__ void __launch_bounds__(256) k_scan_down(F f, NSrc ns, const uint32_t *partials, Out out,
                                                   int64_t *__restrict__ n_total) {
    chain_start();
    __shared__ uint32_t s_w[8];
    uint32_t beg, end;
    block_range(ns.get(), beg, end);
    uint32_t before = 0;                       // the counts of the blocks before this one
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += 256) before += partials[b];
    uint32_t run;
    block_scan_256(before, s_w, &run);
    for (uint32_t t0 = beg; t0 < end; t0 += kSortTile) {
        uint32_t v[kSortItems];
        uint32_t sum = 0;
        const uint32_t i0 = t0 + threadIdx.x * kSortItems;
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            v[k] = (i0 + k < end) ? f(i0 + k) : 0;
            sum += v[k];
        }
        uint32_t tot;
        uint32_t off = run + block_scan_256(sum, s_w, &tot);
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            if (i0 + k < end) out(i0 + k, off, v[k]);
            off += v[k];
        }
        run += tot;
    }
    if (n_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_total = run;   // the last block: the total
}

// --- functors ---
struct KeepFlag {
    const float *cmax;
    float thr;
    __device__ __forceinline__ uint32_t operator()(uint32_t i) const { return cmax[i] >= thr ? 1u : 0u; }
};
struct ActiveFlag {         // keep unless trainable and activity / samples <= thr
    const float *act;
    const uint8_t *layer;
    uint32_t mask;
    float inv_samples, thr;
    __device__ __forceinline__ uint32_t operator()(uint32_t i) const {
        const bool trainable = (mask >> layer[i]) & 1u;
        return (trainable && act[i] * inv_samples <= thr) ? 0u : 1u;
    }
};
struct KeepOut {
    uint8_t *keep;
    int32_t *idx;
    __device__ __forceinline__ void operator()(uint32_t i, uint32_t off, uint32_t v) const {
        keep[i] = static_cast<uint8_t>(v);
        if (v && idx) idx[off] = static_cast<int32_t>(i);
    }
};

// ---------------------------------------------------------------------------
// Depth sort.

struct VisSrc {             // one view: visible where its tile count is non-zero
    const uint32_t *tiles, *depth;
    __device__ __forceinline__ explicit VisSrc(const SortView &v) : tiles(v.tiles), depth(v.depth) {}
    __device__ __forceinline__ bool visible(uint32_t i) const { return tiles[i] > 0; }
    __device__ __forceinline__ uint32_t key(uint32_t i) const { return depth[i]; }
    __device__ __forceinline__ void settle(uint32_t) const {}
};
struct VisSrc2 {            // two eyes: visible to either; keyed by view a's depth where view a sees it
    const uint32_t *tiles_a, *depth_a, *tiles_b, *depth_b;
    Rec *rec_a, *rec_b;
    __device__ __forceinline__ explicit VisSrc2(const SortView &v)
        : tiles_a(v.tiles), depth_a(v.depth), tiles_b(v.tiles_b), depth_b(v.depth_b), rec_a(v.rec), rec_b(v.rec_b) {}
    // A visible Gaussian that one eye does not see is in both eyes' order, but that eye's record of it was not
    // written: an empty tile rectangle there, so its binning passes the Gaussian over.
    __device__ __forceinline__ void settle(uint32_t i) const {
        if (tiles_a[i] == 0) rec_a[i].c.z = rec_a[i].c.w = 0.f;
        if (tiles_b[i] == 0) rec_b[i].c.z = rec_b[i].c.w = 0.f;
    }
    __device__ __forceinline__ bool visible(uint32_t i) const { return tiles_a[i] > 0 || tiles_b[i] > 0; }
    __device__ __forceinline__ uint32_t key(uint32_t i) const { return tiles_a[i] > 0 ? depth_a[i] : depth_b[i]; }
};

constexpr int kLookCounters = 256;                 // one per digit
constexpr uint64_t kLookAgg = 1ull << 32;          // the tile's own count is published
constexpr uint64_t kLookIncl = 2ull << 32;         // the count of every tile up to and including it
constexpr uint32_t kSpinLimit = 1u << 20;
#ifdef GS_DEBUG
// Test hooks of the look-back wait (gs_debug_sort_wait): its iteration limit,
// and a digit kernel whose first tile never publishes its counts.
uint32_t g_dbg_spin_limit = kSpinLimit;
int g_dbg_withhold_pass = -1;
#endif

__device__ __forceinline__ void st_volatile(uint64_t *p, uint64_t v) { *reinterpret_cast<volatile uint64_t *>(p) = v; }
__device__ __forceinline__ uint64_t ld_volatile(const uint64_t *p) {
    return *reinterpret_cast<const volatile uint64_t *>(p);
}

// Digit kernels that run: one per 8-bit digit below the highest bit where the
// smallest and largest visible key differ, and always the first (it also
// compacts the visible Gaussians).
__device__ __forceinline__ int sort_passes(const Ctl *ctl) {
    const uint32_t v = ctl->n_vis > 1 ? (~ctl->depth_mm[0]) ^ ctl->depth_mm[1] : 0u;
    const int m = v ? (39 - __clz(v)) / 8 : 0;     // ceil((32 - clz) / 8)
    return m > 1 ? m : 1;
}

constexpr int kPassThreads = 512;
// Per SM: at most 64 registers.  Without the bound (86) one CTA filled an SM and a kernel ran in five waves of 152
// tiles: sort of 3M 0.115 -> 0.095 ms, of eight times 500,000 0.166 -> 0.117, of 1.2M 0.057 -> 0.049 (540,000 visible of
// 1.2M, which fill one wave: 0.039 -> 0.042); three (40 registers, spilling): 0.102 and 0.125.
constexpr int kPassCtas = 2;
constexpr int kPassWarps = kPassThreads / 32;
constexpr int kPassTile = kPassThreads * kSortItems;
static_assert(kPassTile % kSortTile == 0, "a digit-kernel tile is whole histogram rounds");

// Tile counts of the first digit kernel: cnt[tile][digit] and their sums
// over groups of 2^lg consecutive tiles, grp[group][digit].
struct TileCounts {
    uint32_t *cnt, *grp;
    int lg;
};

// A view's sort with what its kernels derive from the sizes.
struct SortJob {
    SortView v;
    TileCounts tc;
    uint32_t nt;             // tiles of the first digit kernel
    uint32_t spin_limit;     // see SortBufs
    int withhold;
};

// Exclusive prefix of counter c over the tiles before tile t (whose own count
// `own` is already published as an aggregate unless t == 0); publishes the
// inclusive prefix of tile t.  The predecessors are read kLookWindow at a time,
// nearest first, so a walk over tiles that only hold aggregates costs one
// memory latency per window instead of one per tile (windows of eight spill).
constexpr int kLookWindow = 4;
__device__ uint32_t look_back(uint64_t *status, uint32_t t, int c, uint32_t own, Ctl *ctl, uint32_t spin_limit,
                              bool publish) {
    uint32_t excl = 0;
    int64_t j = static_cast<int64_t>(t) - 1;
    uint32_t spins = 0;
    while (j >= 0) {
        uint64_t w[kLookWindow];
#pragma unroll
        for (int k = 0; k < kLookWindow; ++k)
            w[k] = j - k >= 0 ? ld_volatile(status + static_cast<size_t>(j - k) * kLookCounters + c) : kLookIncl;
        int used = 0;
        bool incl = false, waiting = false;
#pragma unroll
        for (int k = 0; k < kLookWindow; ++k) {
            if (incl || waiting) continue;
            const uint64_t flag = w[k] & ~0xFFFFFFFFull;
            if (flag == 0) {
                waiting = true;
                continue;
            }
            excl += static_cast<uint32_t>(w[k]);
            ++used;
            incl = flag == kLookIncl;
        }
        if (incl) break;
        j -= used;
        if (waiting) {
            if (++spins > spin_limit) {
                // What this kernel writes will have holes, keys that the digit histograms do not count: no tile for the
                // kernels after it.  (Asking every CTA for the error status first cost 7 us for 3M Gaussians.)
                ctl->st.error = GS_ERR_TIMEOUT;
                for (int p = 1; p < 4; ++p) atomicOr(&ctl->sort_ticket[p], 0x80000000u);
                break;
            }
            __nanosleep(64);
        }
    }
    if (publish) st_volatile(status + static_cast<size_t>(t) * kLookCounters + c, kLookIncl | (excl + own));
    return excl;
}

// One CTA per tile of the first digit kernel: the visible count, the key
// range, the four digit histograms, and the tile's count of every first digit.
// Four Gaussians per thread: with sixteen the chain of a warp's shuffles and
// votes set the time of small scenes (4,096 Gaussians 12.5 -> 7.8 us, 1.2M 16.5 -> 10.6,
// 3M 24.9 -> 17.1).
constexpr int kHistThreads = 1024;
constexpr int kHistItems = kPassTile / kHistThreads;

template <class Src, int NV>
__global__ void __launch_bounds__(kHistThreads) k_sort_hist(const __grid_constant__ Views<SortJob, NV> B) {
    chain_start();
    __shared__ uint32_t s_h[4][256];
    __shared__ uint32_t s_vis, s_kinv, s_kmax;
    const SortJob &J = B[blockIdx.y];
    const uint32_t n = J.v.n;
    const uint32_t t = blockIdx.x;
    if (t >= J.nt) return;
    const Src src(J.v);
    uint32_t *__restrict__ ghist = J.v.w.ghist;
    Ctl *ctl = J.v.ctl;
    const TileCounts tc = J.tc;
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < 4 * 256; k += kHistThreads) (&s_h[0][0])[k] = 0;
    if (threadIdx.x == 0) s_vis = s_kinv = s_kmax = 0;         // (0 is neutral for both maxima)
    const uint32_t beg = t * kPassTile;
    bool vis[kHistItems];
    uint32_t key[kHistItems];
#pragma unroll
    for (int r = 0; r < kHistItems; ++r) {
        const uint32_t i = beg + r * kHistThreads + threadIdx.x;
        vis[r] = i < n && src.visible(i);
    }
#pragma unroll
    for (int r = 0; r < kHistItems; ++r) key[r] = vis[r] ? src.key(beg + r * kHistThreads + threadIdx.x) : 0u;
    __syncthreads();
    uint32_t kinv = 0, kmax = 0, cnt = 0;
#pragma unroll
    for (int r = 0; r < kHistItems; ++r) {
        if (vis[r]) {
            src.settle(beg + r * kHistThreads + threadIdx.x);
            kinv = max(kinv, ~key[r]);
            kmax = max(kmax, key[r]);
        }
        const unsigned vm = __ballot_sync(FULL, vis[r]);
        if (vm == 0) continue;
        cnt += __popc(vm);
        const int leader = __ffs(vm) - 1;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            // one atomic when the warp's visible keys share the digit (the high digits
            // of depths in a narrow range), else one per key
            const uint32_t d = (key[r] >> (8 * p)) & 255u;
            const uint32_t dl = __shfl_sync(FULL, d, leader);
            if (__all_sync(FULL, !vis[r] || d == dl)) {
                if (lane == leader) atomicAdd(&s_h[p][dl], __popc(vm));
            } else if (vis[r]) {
                atomicAdd(&s_h[p][d], 1u);
            }
        }
    }
    kinv = __reduce_max_sync(FULL, kinv);
    kmax = __reduce_max_sync(FULL, kmax);
    if (lane == 0 && cnt) {
        atomicAdd(&s_vis, cnt);
        atomicMax(&s_kinv, kinv);
        atomicMax(&s_kmax, kmax);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_vis) {
        atomicAdd(&ctl->n_vis, s_vis);
        atomicAdd(&ctl->st.n_visible, s_vis);
        atomicMax(&ctl->depth_mm[0], s_kinv);
        atomicMax(&ctl->depth_mm[1], s_kmax);
    }
    for (int k = threadIdx.x; k < 4 * 256; k += kHistThreads) {
        const uint32_t c = (&s_h[0][0])[k];
        if (c) atomicAdd(&ghist[k], c);
    }
    if (threadIdx.x < 256) {
        const uint32_t c0 = s_h[0][threadIdx.x];
        tc.cnt[static_cast<size_t>(t) * kLookCounters + threadIdx.x] = c0;
        if (c0) atomicAdd(&tc.grp[static_cast<size_t>(t >> tc.lg) * kLookCounters + threadIdx.x], c0);
    }
}

// One digit kernel's buffers: pass p reads what pass p - 1 wrote.
struct SortBufs {
    const uint32_t *kin, *vin;       // digit kernels after the first: this pass's input
    uint32_t *kout, *vout;           // the next digit kernel's input
    uint32_t *final_out;             // Gaussian indices in depth order (last digit kernel)
    uint32_t *vis_index;             // first digit kernel: visible indices in index order
    const uint32_t *ghist;           // [4][256] digit histograms of the visible keys
    TileCounts tc;                   // first digit kernel: tile and group counts
    uint64_t *status, *status_next;  // look-back words [tile][256] of this (after the first) and the next pass
    uint32_t spin_limit;             // iterations a look-back waits for a predecessor before GS_ERR_TIMEOUT
    int withhold;                    // GS_DEBUG test hook: this kernel's first tile publishes nothing (-1: off)
    __device__ __forceinline__ SortBufs(const SortJob &J, int p) {
        const SortWork &w = J.v.w;
        kin = w.keys[(p & 1) ^ 1];
        vin = w.vals[(p & 1) ^ 1];
        kout = w.keys[p & 1];
        vout = w.vals[p & 1];
        final_out = w.order;
        vis_index = w.vis_index;
        ghist = w.ghist;
        tc = J.tc;
        status = w.status + static_cast<size_t>(p - 1) * J.nt * kLookCounters;       // (p > 0)
        status_next = w.status + static_cast<size_t>(p) * J.nt * kLookCounters;      // (p < 3)
        spin_limit = J.spin_limit;
        withhold = J.withhold;
    }
};

// One digit (bits 8 pass .. 8 pass + 7) of the stable LSD sort, on tiles of
// kPassTile items and CTAs of kPassThreads threads.  Warp w ranks the
// contiguous run [256 w, 256 w + 256) of its tile in 8 rounds of 32 with
// warp-private 16-bit digit counters, so items are ranked in index order; the
// tile is then sorted by digit in shared memory and written out in that order,
// so consecutive threads store consecutive addresses of one digit's run.

// The lanes that hold a valid item of the same digit (of valid lanes; the
// others' result is not used): a ballot per bit.  match.any took about 900
// cycles a round with the 16 warps of a CTA (more than half the time of a
// tile), the ballots 250: 3M
// Gaussians 0.147 -> 0.114 ms, eight times 500,000 0.206 -> 0.165, 4,096 0.032 -> 0.026 (all four kernels).
__device__ __forceinline__ unsigned same_digit(uint32_t d, bool valid) {
    unsigned peers = __ballot_sync(FULL, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const unsigned m = __ballot_sync(FULL, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// Exclusive scan over the 512 threads of a block; *total = sum of all v.
__device__ __forceinline__ uint32_t block_scan_512(uint32_t v, uint32_t *s_w, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kPassWarps ? s_w[lane] : 0;
#pragma unroll
        for (int o = 1; o < kPassWarps; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kPassWarps) s_w[lane] = w;
    }
    __syncthreads();
    const uint32_t base = warp > 0 ? s_w[warp - 1] : 0;
    *total = s_w[kPassWarps - 1];
    __syncthreads();
    return base + x - v;
}

template <class Src, bool FIRST, int NV>
__global__ void __launch_bounds__(kPassThreads, kPassCtas) k_sort_pass(const __grid_constant__ Views<SortJob, NV> views, int pass) {
    chain_start();
    __shared__ uint16_t s_wc[kPassWarps][256];   // per-warp digit counts, then per-warp digit bases
    __shared__ uint32_t s_lstart[256];            // start of each digit's run in the locally sorted tile
    __shared__ uint32_t s_off[256];               // global position of each digit's run
    __shared__ uint32_t s_key[kPassTile], s_val[kPassTile];
    __shared__ uint32_t s_w[kPassWarps], s_vw[kPassWarps];
    __shared__ uint32_t s_part[256];               // per digit: its count in this group's tiles before this one
    __shared__ uint32_t s_ticket, s_visbase;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const SortJob &J = views[blockIdx.y];
    Ctl *ctl = J.v.ctl;
    const uint32_t n_all = J.v.n;
    if (blockIdx.x >= J.nt) return;
    const int passes = sort_passes(ctl);
    if (pass >= passes) return;
    const Src src(J.v);
    const SortBufs B(J, FIRST ? 0 : pass);
    const bool last = pass == passes - 1;
    const uint32_t n_vis = min(ctl->n_vis, n_all);
    const uint32_t n = FIRST ? n_all : n_vis;
    const uint32_t ntiles = (n + kPassTile - 1) / kPassTile;
    uint32_t t = blockIdx.x;                       // the first digit kernel: the histogram pass's tiles
    // as many CTAs as tiles take part, the first ones: they start on one SM each before any SM gets a second
    if (t >= ntiles) return;
    if (!FIRST && threadIdx.x == 0) s_ticket = atomicAdd(&ctl->sort_ticket[pass], 1u);
    for (int e = threadIdx.x; e < kPassWarps * 256; e += kPassThreads) (&s_wc[0][0])[e] = 0;
    __syncthreads();
    if (!FIRST) {
        t = s_ticket;
        if (t >= ntiles) return;                   // (a wait of this or an earlier digit kernel ran out)
    }
#ifdef GS_DEBUG
    const bool publish = !(pass == B.withhold && t == 0);
#else
    constexpr bool publish = true;
#endif
    if (!last && t < (n_vis + kPassTile - 1) / kPassTile)
        for (int c = threadIdx.x; c < kLookCounters; c += kPassThreads)
            B.status_next[static_cast<size_t>(t) * kLookCounters + c] = 0;
    const int shift = 8 * pass;
    const uint32_t run0 = t * kPassTile + warp * 256;
    uint32_t key[kSortItems], val[kSortItems], rank[kSortItems], vrank[kSortItems];
    bool valid[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t i = run0 + r * 32 + lane;
        if constexpr (FIRST) {
            valid[r] = i < n && src.visible(i);
            val[r] = i;
        } else {
            valid[r] = i < n;
            val[r] = valid[r] ? B.vin[i] : 0u;
        }
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t i = run0 + r * 32 + lane;
        if constexpr (FIRST) key[r] = valid[r] ? src.key(i) : 0u;
        else key[r] = valid[r] ? B.kin[i] : 0u;
    }
    uint32_t vw = 0;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t d = (key[r] >> shift) & 255u;
        const unsigned peers = same_digit(d, valid[r]);
        const uint32_t before = valid[r] ? s_wc[warp][d] : 0;
        rank[r] = before + __popc(peers & lt);
        __syncwarp();
        if (valid[r] && (peers & lt) == 0) s_wc[warp][d] = static_cast<uint16_t>(before + __popc(peers));
        __syncwarp();
        if constexpr (FIRST) {
            const unsigned vb = __ballot_sync(FULL, valid[r]);
            vrank[r] = vw + __popc(vb & lt);
            vw += __popc(vb);
        }
    }
    if constexpr (FIRST) {
        if (lane == 0) s_vw[warp] = vw;
    }
    __syncthreads();
    const int d = threadIdx.x & 255;
    const bool dig = threadIdx.x < 256;
    uint32_t part = 0;
    if constexpr (FIRST) {
        // the count of digit d in the tiles before this one: the first 256 threads sum the groups before
        // this tile's group, the others the tiles before it in its group
        const uint32_t g0 = t >> B.tc.lg;
        if (dig) {
            const uint32_t *gp = B.tc.grp + d;
#pragma unroll 8
            for (uint32_t g = 0; g < g0; ++g) part += gp[static_cast<size_t>(g) * kLookCounters];
        } else {
            const uint32_t *cp = B.tc.cnt + d;
#pragma unroll 8
            for (uint32_t u = g0 << B.tc.lg; u < t; ++u) part += cp[static_cast<size_t>(u) * kLookCounters];
            s_part[d] = part;
        }
    }
    // per digit d (the first 256 threads): exclusive prefix over the warps, the tile's count, and (after
    // the first digit kernel) its publication
    uint32_t acc = 0;
    if (dig) {
#pragma unroll
        for (int w = 0; w < kPassWarps; ++w) {
            const uint32_t c = s_wc[w][d];
            s_wc[w][d] = static_cast<uint16_t>(acc);
            acc += c;
        }
        if (!FIRST && publish)
            st_volatile(B.status + static_cast<size_t>(t) * kLookCounters + d, (t == 0 ? kLookIncl : kLookAgg) | acc);
    }
    uint32_t ntile;
    const uint32_t ls = block_scan_512(acc, s_w, &ntile);      // synchronises: s_part is complete
    if (dig) s_lstart[d] = ls;
    uint32_t gtot;
    const uint32_t gbase = block_scan_512(dig ? B.ghist[pass * 256 + d] : 0u, s_w, &gtot);
    uint32_t excl = 0;
    if (dig) excl = FIRST ? part + s_part[d] : look_back(B.status, t, d, acc, ctl, B.spin_limit, publish);
    if (dig) s_off[d] = gbase + excl;
    if constexpr (FIRST) {
        // the items of all digits in the tiles before this one are the visible Gaussians before it
        uint32_t before;
        block_scan_512(excl, s_w, &before);
        if (d == 0) s_visbase = before;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        if (valid[r]) {
            const uint32_t dd = (key[r] >> shift) & 255u;
            const uint32_t lpos = s_lstart[dd] + s_wc[warp][dd] + rank[r];
            s_key[lpos] = key[r];
            s_val[lpos] = val[r];
        }
    }
    if constexpr (FIRST) {
        uint32_t vbase = s_visbase;
        for (int w = 0; w < warp; ++w) vbase += s_vw[w];
#pragma unroll
        for (int r = 0; r < kSortItems; ++r)
            if (valid[r]) B.vis_index[vbase + vrank[r]] = val[r];
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < ntile; i += kPassThreads) {
        const uint32_t k = s_key[i];
        const uint32_t dd = (k >> shift) & 255u;
        const uint32_t pos = s_off[dd] + (i - s_lstart[dd]);
        if (!GS_CHECK(pos < n_vis, ctl, kSiteSortScatter)) continue;
        if (last) {
            B.final_out[pos] = s_val[i];
        } else {
            B.kout[pos] = k;
            B.vout[pos] = s_val[i];
        }
    }
}

// The shared order of two eyes: the other eye's visible list and counts, and an error of the sort (a wait that ran out
// leaves the order unfinished, and the other eye bins in it too).
__global__ void __launch_bounds__(256) k_share_order(const Ctl *from, const uint32_t *vis, Ctl *to,
                                                     uint32_t *__restrict__ vis_to, uint32_t n) {
    chain_start();
    const uint32_t nv = from->n_vis;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        to->n_vis = nv;
        to->st.n_visible = from->st.n_visible;
        if (from->st.error != GS_OK) to->st.error = from->st.error;
    }
    for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < min(nv, n); i += gridDim.x * 256u) vis_to[i] = vis[i];
}

// 2^lg tiles per group: the least with 2^(2 lg) >= tiles.
int sort_group_log(uint32_t nt) {
    int lg = 0;
    while ((static_cast<uint64_t>(1) << (2 * lg)) < nt) ++lg;
    return lg;
}

// The jobs of the views that hold Gaussians; returns how many, and the most tiles of one.
int sort_jobs(const SortView *views, int n, SortJob *jobs, uint32_t *most) {
    int m = 0;
    *most = 0;
    for (int i = 0; i < n && m < kMaxBatch; ++i) {
        if (views[i].n <= 0) continue;
        SortJob &j = jobs[m++];
        j.v = views[i];
        j.nt = sort_tiles(views[i].n);
        j.tc.cnt = views[i].w.cnt;
        j.tc.grp = views[i].w.grp;
        j.tc.lg = sort_group_log(j.nt);
#ifdef GS_DEBUG
        j.spin_limit = g_dbg_spin_limit;
        j.withhold = g_dbg_withhold_pass;
#else
        j.spin_limit = kSpinLimit;
        j.withhold = -1;
#endif
        *most = j.nt > *most ? j.nt : *most;
    }
    return m;
}

// f(Src, views) for the two-eye order (a single view) or the views' own.
template <class F>
void with_sort(const SortJob *jobs, int m, F f) {
    if (jobs[0].v.tiles_b) {
        Views<SortJob, 1> b;
        b.v[0] = jobs[0];
        b.n = 1;
        f(static_cast<VisSrc2 *>(nullptr), b);
    } else {
        with_views(jobs, m, [&](const auto &b) { f(static_cast<VisSrc *>(nullptr), b); });
    }
}

template <class Src, int NV>
void hist_kernel(Src *, const Views<SortJob, NV> &b, uint32_t most, cudaStream_t st) {
    // the histograms and the group counts were cleared with the control block
    launch_chained(k_sort_hist<Src, NV>, dim3(most, b.n), kHistThreads, 0, st, b);
}

template <class Src, int NV>
void digit_kernels(Src *, const Views<SortJob, NV> &b, uint32_t most, cudaStream_t st) {
    launch_chained(k_sort_pass<Src, true, NV>, dim3(most, b.n), kPassThreads, 0, st, b, 0);
    for (int p = 1; p < 4; ++p)
        launch_chained(k_sort_pass<Src, false, NV>, dim3(most, b.n), kPassThreads, 0, st, b, p);
}

// ---------------------------------------------------------------------------

}  // namespace

int sort_blocks() {
    static PerDevice cache;
    return cache.get([] {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int g = 4 * (sms > 0 ? sms : 80);
        return g < kMaxSortBlocks ? g : kMaxSortBlocks;
    });
}

uint32_t sort_tiles(int64_t n) { return static_cast<uint32_t>((n + kPassTile - 1) / kPassTile); }

size_t sort_count_bytes(int64_t n) {
    return static_cast<size_t>(sort_tiles(n > 0 ? n : 1)) * kLookCounters * sizeof(uint32_t);
}

size_t sort_status_bytes(int64_t n) {
    return 3 * static_cast<size_t>(sort_tiles(n > 0 ? n : 1)) * kLookCounters * sizeof(uint64_t);
}

size_t sort_group_bytes(int64_t n) {
    // ceil(sqrt(tiles)) groups: never fewer than the ceil(tiles / 2^lg) in use (2^lg >= sqrt(tiles)), and
    // non-decreasing in n, so a workspace sized for n Gaussians also holds any smaller scene
    const uint32_t nt = sort_tiles(n > 0 ? n : 1);
    uint32_t g = 1;
    while (static_cast<uint64_t>(g) * g < nt) ++g;
    return static_cast<size_t>(g) * kLookCounters * sizeof(uint32_t);
}

cudaError_t launch_sort_histograms(const SortView *views, int n, cudaStream_t st) {
    SortJob jobs[kMaxBatch];
    uint32_t most;
    const int m = sort_jobs(views, n, jobs, &most);
    if (m) with_sort(jobs, m, [&](auto *src, const auto &b) { hist_kernel(src, b, most, st); });
    return cudaGetLastError();
}

cudaError_t launch_sort_digits(const SortView *views, int n, cudaStream_t st) {
    SortJob jobs[kMaxBatch];
    uint32_t most;
    const int m = sort_jobs(views, n, jobs, &most);
    if (m) with_sort(jobs, m, [&](auto *src, const auto &b) { digit_kernels(src, b, most, st); });
    return cudaGetLastError();
}

cudaError_t launch_share_order(const Ctl *from, const uint32_t *vis, Ctl *to, uint32_t *vis_to, int n,
                               cudaStream_t st) {
    launch_chained(k_share_order, sort_blocks(), 256, 0, st, from, vis, to, vis_to, static_cast<uint32_t>(n));
    return cudaGetLastError();
}

cudaError_t launch_activity_prune(const float *activity, const uint8_t *layer, uint32_t train_mask, int n,
                                  float samples, float thr, uint8_t *keep, int32_t *keep_index, int64_t *n_keep,
                                  uint32_t *partials, cudaStream_t st) {
    const int G = sort_blocks();
    NSrc ns{nullptr, static_cast<uint32_t>(n)};
    ActiveFlag f{activity, layer, train_mask, 1.f / samples, thr};
    k_scan_reduce<<<G, 256, 0, st>>>(f, ns, partials);
    launch_chained(k_scan_down<decltype(f), KeepOut>, G, 256, 0, st, f, ns, partials, KeepOut{keep, keep_index}, n_keep);
    return cudaGetLastError();
}

cudaError_t launch_prune(const float *contrib_max, int n, float thr, uint8_t *keep, int32_t *keep_index,
                         int64_t *n_keep, uint32_t *partials, cudaStream_t st) {
    const int G = sort_blocks();
    NSrc ns{nullptr, static_cast<uint32_t>(n)};
    KeepFlag f{contrib_max, thr};
    k_scan_reduce<<<G, 256, 0, st>>>(f, ns, partials);
    launch_chained(k_scan_down<decltype(f), KeepOut>, G, 256, 0, st, f, ns, partials, KeepOut{keep, keep_index}, n_keep);
    return cudaGetLastError();
}

}  // namespace gs

extern "C" int gs_debug_sort_wait(uint32_t spin_limit, int32_t withhold_pass) {
#ifdef GS_DEBUG
    if (withhold_pass != -1 && (withhold_pass < 1 || withhold_pass > 3))
        return gs::report(GS_ERR_INVALID, "gs_debug_sort_wait: withhold_pass must be -1 or 1..3");
    gs::g_dbg_spin_limit = spin_limit ? spin_limit : gs::kSpinLimit;
    gs::g_dbg_withhold_pass = withhold_pass;
    return GS_OK;
#else
    (void)spin_limit;
    (void)withhold_pass;
    return gs::report(GS_ERR_INVALID, "gs_debug_sort_wait: only in GS_DEBUG builds");
#endif
}
