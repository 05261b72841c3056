// S2 (second half) - tile binning by two stable bucket passes (Sec. 3.3: the
// splats of each tile are composited in camera-sorted order).
//
// Input: the visible Gaussians in depth order (order[p], p < n_vis, from the
// depth radix sort) and their tile rectangles.  Output: for every tile the
// Gaussians whose rectangle covers it, in depth order (ties by index, as the
// depth sort is stable), concatenated in tile order, and each tile's range.
// That is the stable sort of the (tile, Gaussian) pairs by tile, built
// without sorting the pairs:
//
//  1. Rows.  The (Gaussian, tile row) pairs, in depth order, are split into
//     one list per tile row.  K warps each take a contiguous chunk of the
//     depth order, count its entries per row in shared memory and lay its tile
//     rectangles out in depth order; an exclusive scan over the chunks of every
//     row (row-major count matrices [Ty][K] of entries and of pairs) gives each
//     chunk its place; and a warp per (chunk, 16 rows) writes the entries
//     (Gaussian, x0 | x1 << 16) there, in depth order (emit_group).
//  2. Tiles.  Every row list is cut into pieces of 256 to 1,024 entries
//     (thousands of pieces per frame, so heavy rows spread over all SMs); a
//     warp per piece counts its pairs per tile, a per-row scan over the
//     pieces gives each (piece, tile) its first list position and each tile
//     its range, and a warp per (piece, 16 tiles) writes the Gaussian ids in
//     depth order (emit_group).
//
// Per pair this writes the row entry once (8 B, per row of the rectangle, not
// per tile) and the final Gaussian id once (4 B); the count matrix is a few MB.
// Requires Tx, Ty <= kBinMaxDim (images up to 4096 x 4096).
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// Inclusive warp scan.
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Exclusive scan over a block of NT threads (NT / 32 <= 32 warps).
template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *s_w, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = NT / 32;
    const uint32_t x = warp_incl_scan(v, lane);
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < NW ? s_w[lane] : 0;
        w = warp_incl_scan(w, lane);
        if (lane < NW) s_w[lane] = w;
    }
    __syncthreads();
    const uint32_t base = warp > 0 ? s_w[warp - 1] : 0;
    *total = s_w[NW - 1];
    __syncthreads();
    return base + x - v;
}

// ---- ordered scatter of interval entries ----
//
// A warp streams list entries in order, entry e covering the buckets
// [x0_e, x1_e) and carrying a payload, into kGroup consecutive buckets.  Every
// covered (bucket, entry) pair stores the payload at the bucket's running
// position, so each bucket receives its entries in order:
//   * the entries that reach one of the warp's buckets are compacted, with a
//     bit per bucket they cover;
//   * 32 of them at a time, one per lane, are stored bucket by bucket: a
//     ballot gives the lanes that cover the bucket, a lane's rank is the number
//     of those below it, and they store to consecutive addresses.
// Every lane works on every step and a store instruction covers one or two
// lines.  Bound by instruction issue (67% of the slots).  Per 32 entries the
// scan only tests whether they reach the group and stages them, four words in a
// row; coverage bits are formed for the staged ones.  The tile pass (count,
// scan and write) on the 3M-Gaussian 2064x2208 close view (122M pairs) takes
// 0.398 ms; 0.455 with the coverage formed for every entry and the words taken
// one at a time; 1.043 when pairs were expanded 32 at a time and lanes with
// equal buckets ranked by __match_any_sync or ballots, each 4-byte store a line
// of its own.  Two eyes of a 3M-Gaussian stereo pair (26M pairs each) 0.214,
// 0.244 and 0.472 ms; 1920x1080 (36M pairs) 0.146, 0.166 and 0.307.  Warps that
// take their items from a queue: 0.390 on the close view, but 0.063 against
// 0.052 ms on a 1024x1024 frame.  Also measured: a lane
// per bucket walking the set bits of the transposed coverage matrix (0.490 ms
// on the close view: a third of the lanes idle where the tile lists of a group
// differ in length).
// kGroup: narrower groups compact more often per entry, wider ones leave more
// of a step's lanes without the bucket (0.29 of them store at 16 buckets and
// splats 6.7 tiles wide, 0.17 at 32, 0.45 at 8); 8 took 0.535 ms on the close view.
constexpr int kGroup = 16;

// Bits [a, a + len) (bits at and above 32 fall away).
__device__ __forceinline__ uint32_t bit_run(uint32_t a, uint32_t len) {
    uint32_t m;
    asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(len));
    return m;
}

// The buckets of [c0, c0 + kGroup) that [x0, x1) covers, a bit each.
__device__ __forceinline__ uint32_t coverage(uint32_t x0, uint32_t x1, uint32_t c0) {
    const uint32_t a = static_cast<uint32_t>(max(static_cast<int>(x0 - c0), 0));
    const uint32_t b = static_cast<uint32_t>(max(static_cast<int>(x1 - c0), 0));
    return bit_run(a, b - a) & ((1u << kGroup) - 1u);
}

// Does [x0, x1) = x reach a bucket of [c0, c0 + kGroup)?
__device__ __forceinline__ bool reaches(uint32_t x, uint32_t c0) {
    return (x & 0xFFFFu) < c0 + kGroup && x >= (c0 + 1u) << 16;
}

// Stores one entry per lane (cov: its buckets) at the running positions
// pos[c] of the group's buckets (the same in every lane).
template <class V, class Ok>
__device__ __forceinline__ void emit_group(uint32_t cov, V v, uint32_t (&pos)[kGroup], V *__restrict__ dst,
                                           unsigned lt, Ok ok) {
#pragma unroll
    for (int c = 0; c < kGroup; ++c) {
        const bool in = (cov >> c) & 1u;
        const unsigned b = __ballot_sync(FULL, in);
        const uint32_t p = pos[c] + __popc(b & lt);
        if (in && ok(p)) dst[p] = v;
        pos[c] += __popc(b);
    }
}

// Sum over a warp: three 32-bit reductions, which take 16, 16 and 32 bits of every value without an overflow.
__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
    const uint32_t lo = static_cast<uint32_t>(v);
    return __reduce_add_sync(FULL, lo & 0xFFFFu) + (static_cast<unsigned long long>(__reduce_add_sync(FULL, lo >> 16)) << 16) +
           (static_cast<unsigned long long>(__reduce_add_sync(FULL, static_cast<uint32_t>(v >> 32))) << 32);
}

// Sum over a block of 1024 threads, for thread 0; synchronises the block.
__device__ __forceinline__ unsigned long long block_sum64(unsigned long long v, unsigned long long *s_w) {
    v = warp_sum64(v);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    return threadIdx.x < 32 ? warp_sum64(s_w[threadIdx.x]) : 0ull;
}

// In-place inclusive prefix sum of a[0..n) (shared memory) by one warp.
__device__ __forceinline__ void warp_prefix_inplace(uint32_t *a, int n, int lane) {
    const int per = (n + 31) / 32;
    const int b = min(n, lane * per), e = min(n, b + per);
    uint32_t sum = 0;
    for (int i = b; i < e; ++i) sum += a[i];
    uint32_t run = warp_incl_scan(sum, lane) - sum;
    for (int i = b; i < e; ++i) {
        run += a[i];
        a[i] = run;
    }
    __syncwarp();
}

// The per-row scan of the row pass splits every row's chunk counts (at most
// kBinChunks) into kRowParts parts, one CTA each.
// Gaussians per chunk of the row pass, at least (4,096-Gaussian view 0.019 ms at 32, 0.024 at 128).
constexpr int kChunkMin = 32;
constexpr int kRowParts = 2;
constexpr int kPartChunks = kBinChunks / kRowParts;
constexpr int kPartPerThread = (kPartChunks + 1023) / 1024;
static_assert(kBinChunks % kRowParts == 0, "row-scan part shape");

// Entries per piece of the tile pass (k_bin_rowscan chooses).
constexpr uint32_t kPieceMin = 256, kPieceMax = 1024;
constexpr uint32_t kPieceWarps = 12000;    // (piece, kGroup tiles) items below which pieces stay smaller

struct RowInfo {           // per tile row, in the workspace
    uint32_t start;        // first row-list entry of the row
    uint32_t entries;      // row-list entries of the row
    uint32_t pair_start;   // first pair (final list position) of the row
    uint32_t piece_start;  // first piece of the row (pieces: kPiece-entry parts of row lists)
    uint32_t part_base[kRowParts - 1];   // entries of the row in the chunk parts before parts 1 ..
    uint32_t pad_[5 - kRowParts];        // (32 bytes in all)
};

// The per-row info of a view, and behind it the (entries, pairs) totals of every (row, part) of the row scan.
__device__ __forceinline__ RowInfo *rows_of(const BinView &v) { return static_cast<RowInfo *>(v.rows); }
__device__ __forceinline__ uint2 *part_totals_of(const BinView &v) { return reinterpret_cast<uint2 *>(rows_of(v) + v.Ty); }

// Chunk c of K of the depth order's n entries.
__device__ __forceinline__ void chunk_range(uint32_t n, uint32_t c, uint32_t K, uint32_t &b, uint32_t &e) {
    b = static_cast<uint32_t>(static_cast<uint64_t>(n) * c / K);
    e = static_cast<uint32_t>(static_cast<uint64_t>(n) * (c + 1) / K);
}

// Rows, count: a warp per chunk of the depth order counts its entries and pairs per tile row, and lays the tile
// rectangles out in depth order for the write (x01 and y01: first | last + 1 << 16).
template <int NV>
__global__ void __launch_bounds__(256) k_bin_rows_count(const __grid_constant__ Views<BinView, NV> B) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    const uint32_t *order = V.order;               // (of the kernel before, as M, rows, rowlist and P below: see chain_start)
    const Rec *__restrict__ rec = V.rec;
    uint32_t *__restrict__ M = V.M;
    const Ctl *ctl = V.ctl;
    const uint32_t n_cap = V.n_cap;
    const int Ty = V.Ty;
    __shared__ uint32_t s_cnt[8][kBinMaxDim + 1], s_px[8][kBinMaxDim + 1];
    // an error before the binning (a depth sort that timed out) leaves the order unfinished: do not read it
    if (ctl->st.error != GS_OK) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t K = gridDim.x * 8u;
    uint32_t b, e;
    chunk_range(min(ctl->n_vis, n_cap), blockIdx.x * 8u + warp, K, b, e);
    for (int r = lane; r <= Ty; r += 32) s_cnt[warp][r] = s_px[warp][r] = 0u;
    __syncwarp();
    // ids two groups ahead and records one group ahead of the group being counted, so the gathers overlap
    // the counting of the groups before them
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t gid = b + lane < e ? order[b + lane] : 0u;
    float4 c_nx = b + lane < e ? rec[gid].c : z4;
    gid = b + 32 + lane < e ? order[b + 32 + lane] : 0u;
    for (uint32_t p0 = b; p0 < e; p0 += 32) {
        const float4 cc = c_nx;
        c_nx = p0 + 32 + lane < e ? rec[gid].c : z4;
        gid = p0 + 64 + lane < e ? order[p0 + 64 + lane] : 0u;
        // rows [y0, y1) each get one entry and w pairs: difference array
        const uint32_t r0 = __float_as_uint(cc.z), r1 = __float_as_uint(cc.w);
        if (p0 + lane < e) {
            V.x01[p0 + lane] = (r0 & 0xFFFFu) | (r1 << 16);
            V.y01[p0 + lane] = (r0 >> 16) | (r1 & 0xFFFF0000u);
        }
        const uint32_t y0 = r0 >> 16, y1 = r1 >> 16, w = (r1 & 0xFFFFu) - (r0 & 0xFFFFu);
        if (y1 > y0) {
            atomicAdd(&s_cnt[warp][y0], 1u);
            atomicSub(&s_cnt[warp][y1], 1u);
            atomicAdd(&s_px[warp][y0], w);
            atomicSub(&s_px[warp][y1], w);
        }
    }
    __syncwarp();
    warp_prefix_inplace(s_cnt[warp], Ty, lane);
    warp_prefix_inplace(s_px[warp], Ty, lane);
    __syncthreads();
    // the block's 8 chunks are 8 consecutive columns of the row-major count
    // matrices, written as 32-byte row segments; the pairs matrix follows the
    // entries matrix and is summed per row by the scan
    for (int t = threadIdx.x; t < 8 * Ty; t += blockDim.x) {
        const int r = t >> 3, w = t & 7;
        const size_t at = static_cast<size_t>(r) * K + blockIdx.x * 8u + w;
        M[at] = s_cnt[w][r];
        M[static_cast<size_t>(Ty) * K + at] = s_px[w][r];
    }
}

// Rows, write: a warp per (chunk, kGroup tile rows) writes their row-list entries, as the tile pass does its lists.
// A warp that took all rows of its chunk, 128 Gaussians at a time, stored the 20 or so of them that reach a group of a
// tall image by themselves, two thirds of its lanes idle: row pass of the 3M-Gaussian close view 0.220 -> 0.150 ms,
// stereo pair 0.114 -> 0.100, 1920x1080 0.073 -> 0.062, eight 512x512 views 0.173 -> 0.129.
constexpr int kRowWords = 4;       // words of 32 Gaussians loaded per step, one step ahead

template <int NV>
__global__ void __launch_bounds__(256) k_bin_rows_write(const __grid_constant__ Views<BinView, NV> B, uint32_t K) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    const uint32_t *__restrict__ order = V.order;
    const uint32_t *__restrict__ x01 = V.x01, *__restrict__ y01 = V.y01;
    const uint32_t *M = V.M;
    const RowInfo *rows = rows_of(V);
    uint2 *__restrict__ rowlist = V.rowlist;
    const Ctl *ctl = V.ctl;
    const int Ty = V.Ty;
    constexpr int kBuf = 32 * (kRowWords + 1);
    __shared__ uint2 s_val[8][kBuf];               // Gaussians that reach the warp's rows: a step's and what was left
    __shared__ uint32_t s_rows[8][kBuf];
    if (ctl->st.error != GS_OK) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t n = min(ctl->n_vis, V.n_cap);
    const uint32_t groups = (Ty + kGroup - 1) / kGroup, items = K * groups;
    const auto ok = [&](uint32_t p) { return GS_CHECK(p < ctl->st.dup_capacity, ctl, kSiteRowList); };
    uint2 *val = s_val[warp];
    uint32_t *yy = s_rows[warp];
    for (uint32_t it = blockIdx.x * 8u + warp; it < items; it += gridDim.x * 8u) {
        const uint32_t ch = it / groups, c0 = kGroup * (it - ch * groups);
        uint32_t b, e;
        chunk_range(n, ch, K, b, e);
        if (b >= e) continue;
        uint32_t at = 0;
        if (lane < kGroup && c0 + lane < static_cast<uint32_t>(Ty)) {
            const uint32_t r = c0 + lane, part = ch / (K / kRowParts);
            at = rows[r].start + (part ? rows[r].part_base[part - 1] : 0u) + M[static_cast<size_t>(r) * K + ch];
        }
        uint32_t pos[kGroup];
#pragma unroll
        for (int c = 0; c < kGroup; ++c) pos[c] = __shfl_sync(FULL, at, c);
        uint32_t fill = 0;
        const auto emit = [&](uint32_t k, bool in) {
            const uint32_t y = in ? yy[k + lane] : 0u;
            emit_group(coverage(y & 0xFFFFu, y >> 16, c0), val[k + lane], pos, rowlist, lt, ok);
        };
        uint32_t yn[kRowWords], xn[kRowWords], gn[kRowWords];      // one step ahead
        const auto load = [&](uint32_t p0) {
#pragma unroll
            for (int w = 0; w < kRowWords; ++w) {
                const uint32_t p = p0 + 32 * w + lane;
                const bool in = p < e;
                yn[w] = in ? y01[p] : 0u;
                xn[w] = in ? x01[p] : 0u;
                gn[w] = in ? order[p] : 0u;
            }
        };
        load(b);
        for (uint32_t p0 = b; p0 < e; p0 += 32 * kRowWords) {
            uint32_t y[kRowWords], x[kRowWords], g[kRowWords];
#pragma unroll
            for (int w = 0; w < kRowWords; ++w) {
                y[w] = yn[w];
                x[w] = xn[w];
                g[w] = gn[w];
            }
            load(p0 + 32 * kRowWords);
#pragma unroll
            for (int w = 0; w < kRowWords; ++w) {
                const bool in = reaches(y[w], c0);
                const unsigned km = __ballot_sync(FULL, in);
                if (in) {
                    const uint32_t slot = fill + __popc(km & lt);
                    val[slot] = make_uint2(g[w], x[w]);
                    yy[slot] = y[w];
                }
                fill += __popc(km);
            }
            __syncwarp();
            uint32_t k = 0;
            for (; k + 32 <= fill; k += 32) emit(k, true);
            if (k) {                               // the rest to the front
                const uint2 v = val[k + lane];
                const uint32_t r = yy[k + lane];
                __syncwarp();
                val[lane] = v;
                yy[lane] = r;
                fill -= k;
            }
            __syncwarp();
        }
        if (fill) emit(0, lane < fill);
        __syncwarp();
    }
}

// Per (row, part) (one CTA each, kRowParts parts of K / kRowParts chunks per
// row): exclusive scan of the part's chunk counts in place, and the part's
// entry and pair totals.  The part moves through shared memory with
// coalesced loads and stores (each thread scans a contiguous run of counts);
// the pair total needs only a sum, read coalesced.  The last CTA to finish
// (a counter in the control block) then does the per-row work for the whole
// frame: part bases, row totals, the row, pair and piece starts, and the capacity
// check.  The pair total is added up in 64 bits in the status word: a chunk's pairs of
// a row fit 32 (at most 883,012 Gaussians of 256 tiles), a frame's do not from 65,536
// Gaussians that cover 4096 x 4096 on.  A frame that fits has at most 2^32 - 1 pairs and
// no more entries than pairs, so its starts take 32 bits; after an overflow nothing reads
// them.
template <int NV>
__global__ void __launch_bounds__(1024) k_bin_rowscan(const __grid_constant__ Views<BinView, NV> B, int K) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    uint32_t *__restrict__ M = V.M;
    RowInfo *__restrict__ rows = rows_of(V);
    uint2 *__restrict__ part_tot = part_totals_of(V);
    Ctl *__restrict__ ctl = V.ctl;
    const uint64_t cap = V.cap;
    const int Tx = V.Tx, Ty = V.Ty;
    if (blockIdx.x >= Ty * kRowParts) return;
    __shared__ uint32_t s_w[32];
    __shared__ unsigned long long s_w64[32];
    __shared__ uint32_t s_row[kPartChunks];
    __shared__ bool s_last;
    if (ctl->st.error != GS_OK) return;      // uniform: an error set before this kernel (a sort that timed out)
    const int r = blockIdx.x / kRowParts, part = blockIdx.x % kRowParts;
    const int KP = K / kRowParts;
    uint32_t *row = M + static_cast<size_t>(r) * K + static_cast<size_t>(part) * KP;
    const uint32_t *prow = M + static_cast<size_t>(Ty + r) * K + static_cast<size_t>(part) * KP;   // pairs
    unsigned long long psum = 0;
    for (int i = threadIdx.x; i < KP; i += 1024) {
        s_row[i] = row[i];
        psum += prow[i];
    }
    const unsigned long long ptot = block_sum64(psum, s_w64);      // synchronises the block, so s_row is complete
    uint32_t v[kPartPerThread];
    uint32_t sum = 0;
#pragma unroll
    for (int q = 0; q < kPartPerThread; ++q) {
        const int i = threadIdx.x * kPartPerThread + q;
        v[q] = i < KP ? s_row[i] : 0u;
        sum += v[q];
    }
    uint32_t tot;
    uint32_t run = block_excl_scan<1024>(sum, s_w, &tot);
#pragma unroll
    for (int q = 0; q < kPartPerThread; ++q) {
        const int i = threadIdx.x * kPartPerThread + q;
        if (i < KP) s_row[i] = run;
        run += v[q];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < KP; i += 1024) row[i] = s_row[i];
    if (threadIdx.x == 0) {
        part_tot[blockIdx.x] = make_uint2(tot, static_cast<uint32_t>(ptot));
        atomicAdd(reinterpret_cast<unsigned long long *>(&ctl->st.n_dup), ptot);
        __threadfence();
        s_last = atomicAdd(&ctl->bin_scan_done, 1u) == static_cast<uint32_t>(Ty * kRowParts - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the last CTA: per row (thread r < Ty <= 256) the part bases and totals, then the starts
    const volatile uint2 *pt = part_tot;
    const uint64_t pairs = *const_cast<const volatile uint64_t *>(&ctl->st.n_dup);
    uint32_t ent = 0, prs = 0;
    if (threadIdx.x < Ty) {
        for (int p = 0; p < kRowParts; ++p) {
            const uint32_t e = pt[threadIdx.x * kRowParts + p].x;
            if (p > 0) rows[threadIdx.x].part_base[p - 1] = ent;
            ent += e;
            prs += pt[threadIdx.x * kRowParts + p].y;
        }
        rows[threadIdx.x].entries = ent;
    }
    uint32_t te, tp, tq;
    const bool in = threadIdx.x < Ty;
    const uint32_t s0 = block_excl_scan<1024>(in ? ent : 0u, s_w, &te);
    const uint32_t s1 = block_excl_scan<1024>(in ? prs : 0u, s_w, &tp);
    // entries per piece: the largest that still gives every SM several warps of the scatter (piece, kGroup tiles)
    uint32_t piece = kPieceMin;
    const uint64_t groups = (Tx + kGroup - 1) / kGroup;
    while (piece < kPieceMax && te / (2 * piece) * groups >= kPieceWarps) piece *= 2;
    const uint32_t s2 = block_excl_scan<1024>(in ? (ent + piece - 1) / piece : 0u, s_w, &tq);
    if (in) {
        rows[threadIdx.x].start = s0;
        rows[threadIdx.x].pair_start = s1;
        rows[threadIdx.x].piece_start = s2;
    }
    if (threadIdx.x == 0) {
        ctl->st.dup_capacity = cap;
        ctl->n_pieces = tq;
        ctl->bin_piece = piece;
        if (pairs > cap) ctl->st.error = GS_ERR_WORKSPACE;
    }
}

// The pieces of the row lists.  s_ps[r]: first piece of row r, s_ps[Ty]: their
// number.  Row of piece p: the largest r with s_ps[r] <= p.
__device__ __forceinline__ void load_piece_starts(uint32_t *s_ps, const RowInfo *rows, int Ty, const Ctl *ctl) {
    for (int r = threadIdx.x; r < Ty; r += blockDim.x) s_ps[r] = rows[r].piece_start;
    if (threadIdx.x == 0) s_ps[Ty] = ctl->n_pieces;
    __syncthreads();
}
__device__ __forceinline__ int row_of_piece(const uint32_t *s_ps, int Ty, uint32_t p) {
    int lo = 0, hi = Ty - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_ps[mid] <= p) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Tiles, count: a warp per piece counts its pairs per tile into P[piece][Tx].
template <int NV>
__global__ void __launch_bounds__(256) k_bin_tiles_count(const __grid_constant__ Views<BinView, NV> B) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    const uint2 *rowlist = V.rowlist;
    const RowInfo *__restrict__ rows = rows_of(V);
    uint32_t *__restrict__ P = V.P;
    const Ctl *ctl = V.ctl;
    const int Tx = V.Tx, Ty = V.Ty;
    __shared__ uint32_t s_cnt[8][kBinMaxDim + 1];
    __shared__ uint32_t s_ps[kBinMaxDim + 1];
    if (ctl->st.error != GS_OK) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t npieces = ctl->n_pieces, piece = ctl->bin_piece;
    load_piece_starts(s_ps, rows, Ty, ctl);
    for (uint32_t p = blockIdx.x * 8u + warp; p < npieces; p += gridDim.x * 8u) {
        const int row = row_of_piece(s_ps, Ty, p);
        const RowInfo ri = rows[row];
        const uint32_t e0 = ri.start + (p - s_ps[row]) * piece;
        const uint32_t e1 = min(e0 + piece, ri.start + ri.entries);
        uint32_t *Pp = P + static_cast<size_t>(p) * Tx;
        for (int t = lane; t <= Tx; t += 32) s_cnt[warp][t] = 0u;
        __syncwarp();
        uint2 en_nx = e0 + lane < e1 ? rowlist[e0 + lane] : make_uint2(0u, 0u);   // entries one group ahead
        for (uint32_t q0 = e0; q0 < e1; q0 += 32) {
            const uint2 en = en_nx;
            en_nx = q0 + 32 + lane < e1 ? rowlist[q0 + 32 + lane] : make_uint2(0u, 0u);
            // tiles [x0, x1) each get one pair: difference array
            const uint32_t x0 = en.y & 0xFFFFu, x1 = en.y >> 16;
            if (x1 > x0) {
                atomicAdd(&s_cnt[warp][x0], 1u);
                atomicSub(&s_cnt[warp][x1], 1u);
            }
        }
        __syncwarp();
        warp_prefix_inplace(s_cnt[warp], Tx, lane);
        for (int t = lane; t < Tx; t += 32) Pp[t] = s_cnt[warp][t];
        __syncwarp();
    }
}

// Bucket of a list length for the heaviest-first order of the tiles: a
// logarithmic scale with 16 sub-steps per octave; empty lists go last.
__device__ __forceinline__ int work_bucket(uint32_t w) {
    if (w == 0) return kWorkBuckets - 1;
    const int lz = 31 - __clz(w);
    const uint32_t sub = lz >= 4 ? (w >> (lz - 4)) & 15u : (w << (4 - lz)) & 15u;
    return (kWorkBuckets - 2) - (lz * 16 + static_cast<int>(sub));
}

// A tile row's entries of the order (a CTA of 256 threads, at least as many as a row has tiles): (tile, list start,
// list length, first checkpoint segment).  Ties in no particular order: tiles are independent, so the order changes
// no result.  After an error every list is empty.
__device__ __forceinline__ void order_row(const BinView &V, int r, bool ok, uint32_t *s_first, uint32_t *s_w) {
    const int t = threadIdx.x;
    const size_t tile = static_cast<size_t>(r) * V.Tx + t;
    if (!ok) {
        if (t < V.Tx) V.tile_order[tile] = make_uint4(static_cast<uint32_t>(tile), 0u, 0u, 0u);
        return;
    }
    constexpr int kPer = (kWorkBuckets + 255) / 256;
    uint32_t c[kPer], sum = 0, all;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        c[k] = kPer * t + k < kWorkBuckets ? V.tile_hist[kPer * t + k] : 0u;
        sum += c[k];
    }
    uint32_t run = block_excl_scan<256>(sum, s_w, &all);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (kPer * t + k < kWorkBuckets) s_first[kPer * t + k] = run;
        run += c[k];
    }
    __syncthreads();
    if (t < V.Tx) {
        const uint2 rg = V.ranges[tile];
        const int b = work_bucket(rg.y - rg.x);
        V.tile_order[s_first[b] + atomicAdd(&V.tile_hist[kWorkBuckets + b], 1u)] =
            make_uint4(static_cast<uint32_t>(tile), rg.x, rg.y - rg.x, V.seg_base[tile]);
    }
    __syncthreads();
}
static_assert(kBinMaxDim <= 256, "a row's tiles fit the threads of order_row");

// Tiles, write: a warp per (piece, 16 tiles) writes its Gaussian ids.  P holds
// the first list position of every (piece, tile) (k_bin_tiles_scan).
constexpr int kStepWords = 4;      // words of 32 entries loaded per step, one step ahead

template <int NV>
__global__ void __launch_bounds__(256) k_bin_tiles_write(const __grid_constant__ Views<BinView, NV> B) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    const uint2 *__restrict__ rowlist = V.rowlist;
    const RowInfo *__restrict__ rows = rows_of(V);
    const uint32_t *P = V.P;
    uint32_t *__restrict__ list = V.list;
    const Ctl *ctl = V.ctl;
    const int Tx = V.Tx, Ty = V.Ty;
    __shared__ uint2 s_en[8][32 * (kStepWords + 1)];   // entries that reach the warp's tiles: a step's and what was left
    __shared__ uint32_t s_ps[kBinMaxDim + 1];
    __shared__ uint32_t s_first[kWorkBuckets], s_w[8];
    const bool good = ctl->st.error == GS_OK;
    for (int r = blockIdx.x; r < Ty; r += gridDim.x) order_row(V, r, good, s_first, s_w);
    if (!good) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t npieces = ctl->n_pieces, piece = ctl->bin_piece;
    load_piece_starts(s_ps, rows, Ty, ctl);
    const uint32_t groups = (Tx + kGroup - 1) / kGroup;
    const uint64_t items = static_cast<uint64_t>(npieces) * groups;
    const auto ok = [&](uint32_t at) { return GS_CHECK(at < ctl->st.n_dup, ctl, kSitePairList); };
    for (uint64_t it = blockIdx.x * 8u + warp; it < items; it += gridDim.x * 8u) {
        const uint32_t p = static_cast<uint32_t>(it / groups);
        const uint32_t c0 = kGroup * static_cast<uint32_t>(it - static_cast<uint64_t>(p) * groups), t = c0 + lane;
        const int row = row_of_piece(s_ps, Ty, p);
        uint32_t at = 0, next = 0;                 // next: the tile's position after this piece, where P holds it
        if (lane < kGroup && t < static_cast<uint32_t>(Tx)) {
            const uint32_t *Pp = P + static_cast<size_t>(p) * Tx + t;
            at = Pp[0];
            next = p + 1 < s_ps[row + 1] ? Pp[Tx] : at + 1;
        }
        if (!__any_sync(FULL, next != at)) continue;         // no entry of the piece reaches these tiles
        const RowInfo ri = rows[row];
        const uint32_t e0 = ri.start + (p - s_ps[row]) * piece;
        const uint32_t e1 = min(e0 + piece, ri.start + ri.entries);
        uint32_t pos[kGroup];
#pragma unroll
        for (int c = 0; c < kGroup; ++c) pos[c] = __shfl_sync(FULL, at, c);
        uint32_t fill = 0;
        uint2 *buf = s_en[warp];
        const auto emit = [&](uint32_t k, bool in) {
            const uint2 e = buf[k + lane];
            emit_group<uint32_t>(in ? coverage(e.y & 0xFFFFu, e.y >> 16, c0) : 0u, e.x, pos, list, lt, ok);
        };
        uint2 en_nx[kStepWords];                   // entries one step ahead
        const auto entries = [&](uint32_t q0) {
#pragma unroll
            for (int w = 0; w < kStepWords; ++w)
                en_nx[w] = q0 + 32 * w + lane < e1 ? rowlist[q0 + 32 * w + lane] : make_uint2(0u, 0u);
        };
        entries(e0);
        for (uint32_t q0 = e0; q0 < e1; q0 += 32 * kStepWords) {
            uint2 en[kStepWords];
#pragma unroll
            for (int w = 0; w < kStepWords; ++w) en[w] = en_nx[w];
            entries(q0 + 32 * kStepWords);
#pragma unroll
            for (int w = 0; w < kStepWords; ++w) {
                const bool in = reaches(en[w].y, c0);
                const unsigned km = __ballot_sync(FULL, in);
                if (in) buf[fill + __popc(km & lt)] = en[w];
                fill += __popc(km);
            }
            __syncwarp();
            uint32_t k = 0;
            for (; k + 32 <= fill; k += 32) emit(k, true);
            if (k) {                               // the rest to the front
                const uint2 e = buf[k + lane];     // (k + 32 <= 32 (kStepWords + 1): in the buffer)
                __syncwarp();
                buf[lane] = e;
                fill -= k;
            }
            __syncwarp();
        }
        if (fill) emit(0, lane < fill);
        __syncwarp();
    }
}

// Per row (one CTA of 1024 threads): the threads form S slices of TW tiles
// (TW the power of two at or above Tx, at least 16, so S = 1024 / TW <= 64);
// thread (slice s, tile t) sums the counts of tile t over its share of the
// row's pieces; the slice sums give each tile's total and range; then every
// (piece, tile) count is replaced by its first list position.
//
// The CTA that knows a row's tile ranges also prepares them for the forward
// compositor: the first checkpoint segment of every tile (any disjoint
// placement will do: the row takes its segments from a counter), zeroed
// meeting words of the 8x8 blocks, the count of tiles with a list, and the
// counts of a heaviest-first counting sort of the tiles, whose placement
// follows in k_bin_tiles_write.  A kernel of one CTA that walked all tiles for
// this took 45 us for the 17,800 tiles of a 2064 x 2208 view, 21 for the 8,160
// of 1920 x 1080 and 7 for 64; here it costs 2 to 9 us of the binning.
template <int NV>
__global__ void __launch_bounds__(1024) k_bin_tiles_scan(const __grid_constant__ Views<BinView, NV> B) {
    chain_start();
    const BinView &V = B[blockIdx.y];
    const RowInfo *__restrict__ rows = rows_of(V);
    uint32_t *__restrict__ P = V.P;
    uint2 *__restrict__ ranges = V.ranges;
    const Ctl *ctl = V.ctl;
    const int Tx = V.Tx;
    if (blockIdx.x >= V.Ty) return;
    __shared__ uint32_t s_sum[1024];         // [slice][tile]
    __shared__ uint32_t s_off[kBinMaxDim];
    __shared__ uint32_t s_w[32];
    __shared__ uint32_t s_seg;
    const size_t tile0 = static_cast<size_t>(blockIdx.x) * Tx;
    for (int q = threadIdx.x; q < 8 * Tx; q += 1024) V.qdone[8 * tile0 + q] = 0;   // 4 x 64-bit meeting words per tile
    if (ctl->st.error != GS_OK) return;
    int TW = 16;
    while (TW < Tx) TW <<= 1;
    const int S = 1024 / TW;
    const int r = blockIdx.x;
    const int t = threadIdx.x & (TW - 1), sl = threadIdx.x / TW;
    const RowInfo ri = rows[r];
    const uint32_t piece = ctl->bin_piece, npc = (ri.entries + piece - 1) / piece;
    const uint32_t per = (npc + S - 1) / S;
    const uint32_t p0 = ri.piece_start + min(npc, sl * per), p1 = ri.piece_start + min(npc, (sl + 1) * per);
    uint32_t sum = 0;
    if (t < Tx)
        for (uint32_t p = p0; p < p1; ++p) sum += P[static_cast<size_t>(p) * Tx + t];
    s_sum[sl * TW + t] = sum;
    __syncthreads();
    uint32_t tot = 0, before = 0;
    if (t < Tx)
        for (int q = 0; q < S; ++q) {
            const uint32_t v = s_sum[q * TW + t];
            if (q < sl) before += v;
            tot += v;
        }
    uint32_t all;
    const uint32_t toff = block_excl_scan<1024>(sl == 0 && t < Tx ? tot : 0u, s_w, &all);
    const bool mine = sl == 0 && t < Tx;
    if (mine) s_off[t] = toff;                // tile offsets within the row, read by every slice below
    uint32_t rowsegs;
    const uint32_t soff = block_excl_scan<1024>(mine ? ceil_seg(tot) : 0u, s_w, &rowsegs);
    if (threadIdx.x == 0) s_seg = atomicAdd(&V.tile_hist[2 * kWorkBuckets], rowsegs);
    const uint32_t live = __syncthreads_count(mine && tot != 0);
    if (threadIdx.x == 0 && live) atomicAdd(&V.ctl->live_tiles, live);
    if (t < Tx) {
        const uint32_t base = ri.pair_start + s_off[t];
        if (sl == 0) {
            if (GS_CHECK(base + tot <= ctl->st.n_dup, ctl, kSiteRange)) ranges[tile0 + t] = make_uint2(base, base + tot);
            V.seg_base[tile0 + t] = s_seg + soff;
            atomicAdd(&V.tile_hist[work_bucket(tot)], 1u);
        }
        uint32_t run = base + before;
        // eight counts loaded before any of them is replaced, so the loads overlap instead of each waiting
        // behind the previous store
        constexpr int kB = 8;
        for (uint32_t p = p0; p < p1; p += kB) {
            uint32_t v[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) v[k] = p + k < p1 ? P[static_cast<size_t>(p + k) * Tx + t] : 0u;
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                if (p + k < p1) P[static_cast<size_t>(p + k) * Tx + t] = run;
                run += v[k];
            }
        }
    }
}

}  // namespace

cudaError_t launch_bin_rows(const BinView *views, int n, cudaStream_t st) {
    int Ty = 0;
    uint32_t most = 0;
    for (int i = 0; i < n; ++i) {
        if (views[i].Ty > kBinMaxDim || views[i].Tx > kBinMaxDim) return cudaErrorInvalidValue;
        Ty = max(Ty, views[i].Ty);
        most = max(most, views[i].n_cap);
    }
    // chunks of at least kChunkMin Gaussians (a chunk has a column of counts to scan)
    const int blocks = max(min(kBinBlocks, static_cast<int>(most / (8 * kChunkMin))), 1);
    with_views(views, n, [&](const auto &b) {
        constexpr int NV = sizeof(b.v) / sizeof(BinView);
        launch_chained(k_bin_rows_count<NV>, dim3(blocks, n), 256, 0, st, b);
        launch_chained(k_bin_rowscan<NV>, dim3(Ty * kRowParts, n), 1024, 0, st, b, 8 * blocks);
        const int groups = (Ty + kGroup - 1) / kGroup;             // a warp per (chunk, group of rows)
        launch_chained(k_bin_rows_write<NV>, dim3(min(blocks * groups, max(4 * sort_blocks() / n, 1)), n), 256, 0, st, b,
                       8u * blocks);
    });
    return cudaGetLastError();
}

cudaError_t launch_bin_tiles(const BinView *views, int n, cudaStream_t st) {
    int Ty = 0;
    for (int i = 0; i < n; ++i) Ty = max(Ty, views[i].Ty);
    // 16 CTAs per SM, several waves: pieces differ in pairs (half as many: 3% slower)
    const int G = max(sort_blocks() / 4, 4 * sort_blocks() / n);
    with_views(views, n, [&](const auto &b) {
        constexpr int NV = sizeof(b.v) / sizeof(BinView);
        launch_chained(k_bin_tiles_count<NV>, dim3(G, n), 256, 0, st, b);
        launch_chained(k_bin_tiles_scan<NV>, dim3(Ty, n), 1024, 0, st, b);
        launch_chained(k_bin_tiles_write<NV>, dim3(G, n), 256, 0, st, b);
    });
    return cudaGetLastError();
}

size_t bin_piece_bytes(int64_t dup_cap, int Tx, int Ty) {
    // A row list of E entries has ceil(E / piece) pieces of at least kPieceMin entries and the row lists hold at
    // most dup_cap entries, so dup_cap / kPieceMin + Ty rows of counts always suffice; the size grows with the
    // capacity.
    return (static_cast<size_t>(dup_cap) / kPieceMin + Ty + 1) * Tx * 4;
}

// The RowInfo of every row, then the (entries, pairs) totals of every (row, part) of the row scan.
size_t bin_rows_bytes(int Ty) {
    return static_cast<size_t>(Ty) * sizeof(RowInfo) + static_cast<size_t>(Ty) * kRowParts * sizeof(uint2);
}
static_assert(sizeof(RowInfo) == 32, "RowInfo layout");

}  // namespace gs
