// S3 / S4a - front-to-back compositing of each 16x16 tile over its sorted
// splat list (Sec. 3.3: Gaussians rendered as splats in camera-sorted order),
// and its exact backward with the per-Gaussian blend weight alpha*T that
// drives contribution pruning (Sec. 3.2.2).
//
// Work decomposition (compositing is FP32 FMA + MUFU work, not a dense
// contraction, so no tensor cores are involved):
//  * Forward: persistent warps take work items (tile, 8x4 or 8x8 pixel block)
//    from per-view device queues in heaviest-first tile order (the views of a
//    batch in turn) and composite one or two pixels per lane until the block's
//    pixels are done.  The walk goes segment by segment (kSeg list
//    positions), each segment blended from a local product that the
//    transmittance at its start scales; at every segment boundary the warp
//    stores each pixel's transmittance as a checkpoint, with the colour
//    blended from there to the end of the pixel's walk (filled in when the
//    walk ends).
//  * Both passes drop, a chunk of records at a time, the splats that provably stay
//    below alpha = 1/255 over the warp's whole pixel block (see
//    splat_reaches_block); list positions are kept, so nothing changes.
//  * Backward: the blended prefix of a pixel can be thousands of splats long,
//    and walking it serially would make the longest pixel the critical path
//    of the whole kernel.  The checkpoints cut every 8x8 block's walk into
//    segments of at most kSeg positions; persistent warps take (tile, block,
//    segment) items from a queue and each walks its segment back to front
//    from the checkpoint at the segment's end.  The forward writes the items:
//    the second 8x4 block of an 8x8 block to finish knows the block's longest
//    blended prefix, so no ordering pass runs between the two.
//
// splat_alpha() defines the per-(pixel, splat) alpha of both passes; every
// operation is explicitly rounded, and the backward does the same operations on
// two pixels at a time (packed instructions round each half alike), so it
// reproduces the forward's skip decisions bit for bit.
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

constexpr int kFwdThreads = 128;
constexpr int kBwdThreads = 128;
// The backward takes two pixels per lane (an 8x8 block per warp).  Four (16x8) halved the per-splat reduction and
// atomics per pixel but needed 96 registers and culled on a coarser block: 1.2M-Gaussian frame 0.403 ms against 0.362.

// 1/x to about 1 ulp (the hardware reciprocal approximation; x = 1 - alpha is in [0.01, 1]).
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// alpha = min(0.99, o * 2^(A2 (dx + beta dy)^2 + G2 dy^2)), d = pixel - mean.
// Returns alpha; p, dy, ex (= 2^e) and the unclamped product ao are outputs.
__device__ __forceinline__ float splat_alpha(float px, float py, const float4 a, const float4 b, float &p, float &dy,
                                             float &ex, float &ao) {
    const float dx = __fsub_rn(px, a.x);
    dy = __fsub_rn(py, a.y);
    p = __fmaf_rn(a.w, dy, dx);
    const float e = __fmaf_rn(__fmul_rn(a.z, p), p, __fmul_rn(__fmul_rn(b.x, dy), dy));
    ex = ex2_approx(e);
    ao = __fmul_rn(b.y, ex);
    return fminf(kAlphaMax, ao);
}

// Can the splat reach alpha >= 1/255 at some pixel centre of the block
// [x0, x1] x [y0, y1]?  The exponent A2 p^2 + G2 dy^2 (p = dx + beta dy) is a
// sum of two non-positive terms, so max(A2 p^2) + max(G2 dy^2) over the block
// bounds it from above; p is linear, so its range over the block comes from
// the corners.  The test keeps a splat unless even that bound, raised by a
// margin far above single-precision rounding of the per-pixel exponent, gives
// alpha < 1/255: a dropped splat is one the per-pixel test would skip at every
// pixel of the block, so dropping it changes no result.
__device__ __forceinline__ bool splat_reaches_block(const float4 a, const float4 b, float x0, float x1, float y0,
                                                    float y1) {
    const float dylo = y0 - a.y, dyhi = y1 - a.y;
    const float mdy = dylo > 0.f ? dylo : (dyhi < 0.f ? -dyhi : 0.f);
    const float blo = a.w * dylo, bhi = a.w * dyhi;
    const float plo = (x0 - a.x) + fminf(blo, bhi), phi = (x1 - a.x) + fmaxf(blo, bhi);
    const float mp = plo > 0.f ? plo : (phi < 0.f ? -phi : 0.f);
    const float emax = a.z * mp * mp + b.x * mdy * mdy;
    return b.y * ex2_approx(emax + 1e-3f) >= kAlphaMin;
}

__device__ __forceinline__ void load_geo(const Geo *g, float4 &a, float4 &b) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(g));
}

// A splat of the backward's walk: what the block test needs, the blue channel and the layer.
struct Chunk {
    float4 a, b;
    float c;
    uint32_t g, ly;
};

// The splat of an id loaded one chunk earlier: list and record loads of a
// chunk are issued a chunk apart, so the record load does not wait on the
// list load in the same iteration.  n, ctl: the Gaussian count and the bounds
// check of GS_DEBUG builds (nothing in release builds).
__device__ __forceinline__ void fetch_splat(const Geo *__restrict__ geo, const Rec *__restrict__ rec,
                                            const uint8_t *__restrict__ layer, uint32_t g, bool valid, Chunk &ch,
                                            uint32_t n, const Ctl *ctl) {
    if (!valid) return;
    if (!GS_CHECK(g < n, ctl, kSiteBwdId)) {
        ch = Chunk{};              // an inert splat (opacity 0): no block keeps it
        return;
    }
    ch.g = g;
    load_geo(geo + g, ch.a, ch.b);
    ch.c = rec[g].c.x;
    ch.ly = layer[g];
}

struct FwdBatch {
    FwdJob job[kMaxBatch];
    int n;
};

// Forward compositing, segment by segment.  A pixel's walk is cut at the
// checkpoint segments (kSeg list positions).  In every segment the pixel
// blends from a local product P = 1: the colour D it blends there is relative
// to Ts, its transmittance at the segment's start, and the segment ends with
// colour Ts * D and transmittance Ts * P.  The stop test of a splat is
// Ts * P * (1 - alpha) < kTMin, the paper's T < 1e-4 on this factorisation.
// The checkpoints store Ts and the colour blended from the segment on, which
// is all the backward needs to start a segment's walk from its end.
//
// What bounds it, and what the kernel does about it:
//  * A view whose longest walks set its time (up to about 1.5 Mpixels) waits
//    on latencies.  One pixel per lane, and
//    - the kept splats of a chunk are blended kFwdStep at a time: a step
//      computes its alphas together and only the blends form a chain (a splat
//      cost a lone warp 250 cycles of load, exponent, exponential and branch
//      latency one at a time, 67 in steps of four);
//    - chunks of 128 entries, four per lane, so that the records of the next
//      chunk (about 700 cycles from L2) are on their way for as long as four
//      32-entry chunks take to blend;
//    - an item's successor is taken, and its tile's descriptor loaded, while
//      the item is walked, and the exchange of the 8x4 blocks' prefixes is
//      settled behind the next item's first loads: an item used to begin and
//      end with about 2,500 cycles each of dependent L2 accesses;
//    - tiles without a list are one item each, not eight.
//  * Larger launches are bound by instruction issue and by the shared-memory /
//    L1 pipe, where each gathered record costs a cycle per lane and load.  Two
//    pixels per lane (8x8 blocks) halve the gathers, the tests and the items
//    per pixel, and a record's geometry comes in one aligned 32-byte load (Geo);
//    only kept entries fetch their last word (blue), by cp.async.
// Measured (compositing stage, one at a time with 32-entry chunks before):
// 1.2M-Gaussian 1024x1024 frame 0.154 -> 0.114 ms, 1.5M-Gaussian 1037x771 view
// 0.177 -> 0.096, 500k-Gaussian 512x512 view 0.071 -> 0.053, 40k-Gaussian 397x243
// view 0.061 -> 0.040; 3M-Gaussian 2064x2208 view 0.668 -> 0.452, both eyes of the
// stereo pair 0.619 -> 0.380, 1920x1080 view 0.351 -> 0.211.
constexpr int kFwdWarps = kFwdThreads / 32;
constexpr int kFwdStep = 4;
// A warp takes its next item before it walks the current one only where that
// tile's list is at most this long: tiles come heaviest first, so what a
// warp holds back is short too (taken early everywhere, the 1024x1024 frame took
// 0.128 ms instead of 0.114).
constexpr uint32_t kAheadLen = 1024;

template <int PER>
struct FwdKept {            // a chunk's entries that can reach the warp's block
    float4 a[32 * PER + kFwdStep];     // u, v, A2, beta
    float4 b[32 * PER + kFwdStep];     // G2, opacity, r, g
    float blue[32 * PER + kFwdStep];   // (arrives by cp.async)
    uint32_t pos[32 * PER];            // list position
};
template <int PER>
struct FwdSmem {
    FwdKept<PER> kept[kFwdWarps][2];
};

struct FwdLane {        // one pixel's walk
    float Ts;           // transmittance at the start of the current segment
    float P;            // product of (1 - alpha) over the splats blended in the segment
    float D0, D1, D2;   // colour blended in the segment, relative to Ts
    uint32_t last;      // 1 + list position (from the tile's first entry) of the last blended splat
    uint32_t nb;        // blended splats
    bool done;          // stopped (or outside the image)
};

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One tile list's entries on their way to a warp.
template <int PER>
struct FwdStream {
    static constexpr uint32_t kChunk = 32 * PER;
    const uint32_t *list;   // the tile's first entry
    const Geo *geo;
    const Rec *rec;
    uint32_t len;
    float4 a[PER], b[PER];    // this lane's entries of the next chunk
    uint32_t cur[PER];     // their ids
    uint32_t id[PER];      // this lane's ids of the chunk after it
    uint32_t n;             // Gaussian count and status (bounds check of GS_DEBUG builds)
    const Ctl *ctl;

    __device__ __forceinline__ void load_ids(uint32_t pos, int lane) {
#pragma unroll
        for (int k = 0; k < PER; ++k) id[k] = pos + 32 * k + lane < len ? list[pos + 32 * k + lane] : 0u;
    }
    // Loads the entries of the chunk at `pos` (their ids are in id) and the ids of the chunk after it.
    __device__ __forceinline__ void request(uint32_t pos, int lane) {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            cur[k] = id[k];
            if (pos + 32 * k + lane >= len) continue;
            if (GS_CHECK(id[k] < n, ctl, kSiteFwdId)) {
                load_geo(geo + id[k], a[k], b[k]);
            } else {                                // an inert splat (opacity 0): no block keeps it
                a[k] = b[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        load_ids(pos + kChunk, lane);
    }
};

// Blends the kept entries [k, k + S) into the segment state of the lane's pixels
// (PX of them, four rows apart), in order.
template <int S, int PX, int PER>
__device__ __forceinline__ void blend_step(const FwdKept<PER> &K, int k, float px, float py, FwdLane (&L)[PX],
                                           bool (&mine)[PX], int (&lastk)[PX]) {
    float al[S][PX];
    float2 rg[S];
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const float4 a = K.a[k + j], b = K.b[k + j];
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            float p, dy, ex, ao;
            al[j][i] = splat_alpha(px, py + 4.f * i, a, b, p, dy, ex, ao);
        }
        rg[j] = make_float2(b.z, b.w);
    }
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const float bl = K.blue[k + j];
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            const bool act = al[j][i] >= kAlphaMin && !mine[i];
            const float Pn = __fmul_rn(L[i].P, __fsub_rn(1.f, al[j][i]));
            const bool stop = __fmul_rn(L[i].Ts, Pn) < kTMin;
            const float w = __fmul_rn(al[j][i], L[i].P);
            mine[i] = mine[i] || (act && stop);
            if (act && !stop) {
                L[i].D0 = __fmaf_rn(rg[j].x, w, L[i].D0);
                L[i].D1 = __fmaf_rn(rg[j].y, w, L[i].D1);
                L[i].D2 = __fmaf_rn(bl, w, L[i].D2);
                L[i].P = Pn;
                lastk[i] = k + j;
                ++L[i].nb;
            }
        }
    }
}

// Takes the chunk at `pos` of the block at (bx0, by0) (8 x 4 PX pixel centres):
// every lane tests its entries against the block, and those that can
// reach it are staged in K in list order, their blue on its way.  Returns how
// many; requests the chunk after.
template <int PX, int PER>
__device__ __forceinline__ int stage_chunk(FwdStream<PER> &st, uint32_t pos, float bx0, float by0, int lane,
                                           FwdKept<PER> &K) {
    bool keep[PER];
    unsigned km[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        keep[k] = pos + 32 * k + lane < st.len &&
                  splat_reaches_block(st.a[k], st.b[k], bx0, bx0 + 7.f, by0, by0 + (4.f * PX - 1.f));
        km[k] = __ballot_sync(FULL, keep[k]);
    }
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (keep[k]) {
            const int slot = cnt + __popc(km[k] & ((1u << lane) - 1u));
            K.a[slot] = st.a[k];
            K.b[slot] = st.b[k];
            K.pos[slot] = pos + 32 * k + lane;
            cp_async4(&K.blue[slot], &st.rec[st.cur[k]].c.x);
        }
        cnt += __popc(km[k]);
    }
    if (lane < kFwdStep) {                         // inert splats (opacity 0) fill the last step
        K.a[cnt + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        K.b[cnt + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    cp_async_commit();
    st.request(pos + 32 * PER, lane);
    return cnt;
}

// Blends a staged chunk into every lane's pixels.
template <int PX, int PER>
__device__ __forceinline__ void blend_chunk(const FwdKept<PER> &K, int cnt, float px, float py, FwdLane (&L)[PX]) {
    bool mine[PX];
    int lastk[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        mine[i] = L[i].done;
        lastk[i] = -1;
    }
    int k = 0;
    for (; k + kFwdStep / 2 < cnt; k += kFwdStep) blend_step<kFwdStep>(K, k, px, py, L, mine, lastk);
    if (k < cnt) blend_step<kFwdStep / 2>(K, k, px, py, L, mine, lastk);
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        if (lastk[i] >= 0) L[i].last = K.pos[lastk[i]] + 1;    // position of the chunk's last blend, read once
        L[i].done = mine[i];
    }
}

// The live view after v in turn (live != 0, v < 31).
__device__ __forceinline__ int next_live(uint32_t live, int v) {
    const uint32_t after = live & ~((2u << v) - 1u);
    return __ffs(after ? after : live) - 1;
}

// The views of a batch are taken in turn, each from its own heaviest-first queue, so the heaviest blocks of
// every view start first; a view whose queue has run out leaves the rotation.  A view's queue is one 64-bit word,
// (tiles with a list << 32 | items taken): its items are the 8 / PX blocks of every tile with a list, then the
// empty tiles, each as a whole.
template <int PX>
struct FwdQueue {
    static constexpr uint32_t kBlocks = 8 / PX;      // items of a tile with a list
    const FwdBatch &batch;
    uint32_t live;
    int lane;
    __device__ __forceinline__ unsigned long long take(int v) const {      // lane 0's result counts
        return lane == 0 ? atomicAdd(reinterpret_cast<unsigned long long *>(batch.job[v].queue), 1ull) : 0ull;
    }
    // The item taken as q from view v, or from a later live view when v had none left; false: all have run out.
    __device__ __forceinline__ bool resolve(unsigned long long q, int &v, uint32_t &local, uint32_t &tiles) {
        if (lane == 0) {
            for (;;) {
                const uint32_t nl = static_cast<uint32_t>(q >> 32);
                if (static_cast<uint32_t>(q) < (kBlocks - 1u) * nl + static_cast<uint32_t>(batch.job[v].Tn)) break;
                live &= ~(1u << v);
                if (!live) break;
                v = next_live(live, v);
                q = take(v);
            }
        }
        live = __shfl_sync(FULL, live, 0);
        if (!live) return false;
        v = __shfl_sync(FULL, v, 0);
        local = __shfl_sync(FULL, static_cast<uint32_t>(q), 0);
        tiles = __shfl_sync(FULL, static_cast<uint32_t>(q >> 32), 0);
        return true;
    }
};

// The two 8x4 blocks of an 8x8 block meet in one 64-bit word, a half each for (longest blended prefix + 1).  The
// second to arrive knows the 8x8 block's longest blended prefix: it stores it for the backward and appends the
// block's backward work items, one per kSeg positions of the prefix.  They come out in the order the forward
// finishes them, the heaviest tiles last; the backward takes them from the end.  The exchange is sent at the end
// of an item and settled while the next item's records are on their way.
struct FwdMeet {
    unsigned long long old;    // lane 0: the word before this block's half was set
    uint32_t tile, qd, half, prefix;
    int v;
    bool open;
    __device__ __forceinline__ void settle(const FwdBatch &batch, int lane) {
        if (!open) return;
        open = false;
        const FwdJob &J = batch.job[v];
        uint32_t nsg = 0, ibase = 0;
        if (lane == 0) {
            const uint32_t other = static_cast<uint32_t>(old >> (32u * (half ^ 1u)));
            if (other) {
                const uint32_t qm = max(other - 1u, prefix);
                J.qwork[4 * tile + qd] = qm;
                nsg = ceil_seg(qm);
                if (nsg) ibase = atomicAdd(J.n_items, nsg);
            }
        }
        nsg = __shfl_sync(FULL, nsg, 0);
        if (nsg == 0) return;
        ibase = __shfl_sync(FULL, ibase, 0);
        for (uint32_t sg = lane; sg < nsg; sg += 32) J.items[ibase + sg] = make_uint2(tile, (qd << 24) | sg);
    }
};

template <int PX, int PER>
__global__ void __launch_bounds__(kFwdThreads) k_composite_fwd(const __grid_constant__ FwdBatch batch) {
    chain_start();
    extern __shared__ __align__(16) unsigned char s_raw[];
    FwdSmem<PER> &sm = *reinterpret_cast<FwdSmem<PER> *>(s_raw);
    constexpr uint32_t kChunk = 32 * PER, B = FwdQueue<PX>::kBlocks;
    static_assert(kSeg % kChunk == 0, "segments are whole chunks");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    FwdQueue<PX> fq{batch, (1u << batch.n) - 1u, lane};
    FwdMeet meet;
    meet.open = false;
    FwdStream<PER> st;
    int v = static_cast<int>((blockIdx.x * kFwdWarps + warp) % static_cast<uint32_t>(batch.n));
    uint32_t local, tiles;
    bool have = fq.resolve(fq.take(v), v, local, tiles);
    uint4 d = make_uint4(0u, 0u, 0u, 0u);
    const auto slot_of = [](uint32_t l, uint32_t nl) { return l < B * nl ? l / B : l - (B - 1u) * nl; };
    if (have) d = batch.job[v].order[slot_of(local, tiles)];
    const auto take_next = [&](unsigned long long q, int nv) {
        v = nv;
        have = fq.resolve(q, v, local, tiles);
        if (have) d = batch.job[v].order[slot_of(local, tiles)];
    };
    while (have) {
        const FwdJob &J = batch.job[v];
        const int W = J.W, H = J.H, Tx = J.Tx;
        const int tile = static_cast<int>(d.x), ty = tile / Tx, tx = tile - ty * Tx;
        const bool empty = local >= B * tiles;
        const size_t plane = static_cast<size_t>(W) * H;
        if (empty) {
            // no list: the background over the whole tile, 8 pixels per lane; the next item is taken first
            int nv = next_live(fq.live, v);
            const unsigned long long q = fq.take(nv);
            const float3 bg = J.bg;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int x = tx * kTile + (lane & 15), y = ty * kTile + 2 * k + (lane >> 4);
                if (x < W && y < H) {
                    const size_t pix = static_cast<size_t>(y) * W + x;
                    J.image[pix] = bg.x;
                    J.image[plane + pix] = bg.y;
                    J.image[2 * plane + pix] = bg.z;
                    if (J.alpha) J.alpha[pix] = 0.f;
                    J.t_final[pix] = 1.f;
                    J.n_contrib[pix] = 0u;
                }
            }
            take_next(q, nv);
            continue;
        }
        const uint32_t len = d.z;
        st.list = J.list + d.y;
        st.geo = J.geo;
        st.rec = J.rec;
        st.len = len;
        st.n = J.n;
        st.ctl = J.ctl;
        st.load_ids(0, lane);
        cp_async_wait<0>();                             // what the item before had staged beyond its stop
        __syncwarp();
        const int sub = local % B;                      // block column sub & 1, block row sub >> 1
        const int ox = (sub & 1) * 8, oy = (sub >> 1) * 4 * PX;
        const float bx0 = tx * kTile + ox + 0.5f, by0 = ty * kTile + oy + 0.5f;
        const int lx = ox + (lane & 7), ly = oy + (lane >> 3);
        const int x = tx * kTile + lx, y = ty * kTile + ly;
        FwdLane L[PX];
        float C0[PX], C1[PX], C2[PX];                   // colour of the last finished segment
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            L[i] = FwdLane{1.f, 1.f, 0.f, 0.f, 0.f, 0u, 0u, !(x < W && y + 4 * i < H)};
            C0[i] = C1[i] = C2[i] = 0.f;
        }
        const auto all_done = [&]() {
            bool d = L[0].done;
#pragma unroll
            for (int i = 1; i < PX; ++i) d = d && L[i].done;
            return __all_sync(FULL, d) != 0;
        };
        float4 *ck0 = J.ckpt + static_cast<size_t>(d.w) * kTilePix + ly * kTile + lx;
        st.request(0, lane);
        // a short walk: the next item is taken now and its descriptor loaded at the end
        const bool ahead = len <= kAheadLen;
        int nv = next_live(fq.live, v);
        unsigned long long q = 0;
        if (ahead) q = fq.take(nv);
        if constexpr (PX == 1) meet.settle(batch, lane);
        // chunk by chunk, each staged before the one ahead of it is blended
        uint32_t sd = 0;
        int cnt_prev = 0;
        if (!all_done()) {
            for (uint32_t pos = 0, buf = 0;; pos += kChunk, buf ^= 1) {
                const bool more = pos < len;
                int cnt = 0;
                if (more) cnt = stage_chunk<PX>(st, pos, bx0, by0, lane, sm.kept[warp][buf]);
                if (pos > 0) {
                    if (more) cp_async_wait<1>(); else cp_async_wait<0>();
                    __syncwarp();
                    blend_chunk(sm.kept[warp][buf ^ 1], cnt_prev, x + 0.5f, y + 0.5f, L);
                    const bool stop = all_done() || !more;
                    if (stop || pos % kSeg == 0) {
                        // the segment ends: its colour, the transmittance at the next segment's start
#pragma unroll
                        for (int i = 0; i < PX; ++i) {
                            C0[i] = __fmul_rn(L[i].Ts, L[i].D0);
                            C1[i] = __fmul_rn(L[i].Ts, L[i].D1);
                            C2[i] = __fmul_rn(L[i].Ts, L[i].D2);
                            L[i].Ts = __fmul_rn(L[i].Ts, L[i].P);
                            L[i].P = 1.f;
                            L[i].D0 = L[i].D1 = L[i].D2 = 0.f;
                        }
                        if (stop) break;
                        ++sd;
                        if (!GS_CHECK(d.w + sd < J.n_segs, J.ctl, kSiteCkpt)) {
                            --sd;
                            break;
                        }
                        // checkpoint sd: (T at the segment's start, colour of segment sd - 1); rewritten below
#pragma unroll
                        for (int i = 0; i < PX; ++i)
                            ck0[static_cast<size_t>(sd) * kTilePix + 4 * kTile * i] =
                                make_float4(L[i].Ts, C0[i], C1[i], C2[i]);
                    }
                    __syncwarp();                  // the chunk has been read: its buffer is staged next
                }
                cnt_prev = cnt;
            }
        }
        const int mv = v;
        if (ahead) take_next(q, nv);
        else q = fq.take(nv);
        // Checkpoint s holds (T at segment start, colour of segment s-1) as written
        // above; rewrite it, deepest segment first, to (T at segment start, F_s),
        // F_s = colour blended at list positions >= s kSeg.  F_0 is the pixel's colour.
        // Four are read ahead of the chain.
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            float4 *ck = ck0 + 4 * kTile * i;
            for (uint32_t s = sd; s > 0;) {
                float4 raw[4];
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    if (k < s) raw[k] = ck[static_cast<size_t>(s - k) * kTilePix];
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) {
                    if (k >= s) continue;
                    ck[static_cast<size_t>(s - k) * kTilePix] = make_float4(raw[k].x, C0[i], C1[i], C2[i]);
                    C0[i] = __fadd_rn(raw[k].y, C0[i]);
                    C1[i] = __fadd_rn(raw[k].z, C1[i]);
                    C2[i] = __fadd_rn(raw[k].w, C2[i]);
                }
                s = s > 4 ? s - 4 : 0;
            }
            if (x < W && y + 4 * i < H) {
                const size_t pix = static_cast<size_t>(y + 4 * i) * W + x;
                J.image[pix] = __fmaf_rn(L[i].Ts, J.bg.x, C0[i]);
                J.image[plane + pix] = __fmaf_rn(L[i].Ts, J.bg.y, C1[i]);
                J.image[2 * plane + pix] = __fmaf_rn(L[i].Ts, J.bg.z, C2[i]);
                if (J.alpha) J.alpha[pix] = 1.f - L[i].Ts;
                J.t_final[pix] = L[i].Ts;
                J.n_contrib[pix] = L[i].last;
            }
        }
        uint32_t last = L[0].last, nb = L[0].nb;
#pragma unroll
        for (int i = 1; i < PX; ++i) {
            last = max(last, L[i].last);
            nb += L[i].nb;
        }
        meet.prefix = __reduce_max_sync(FULL, last);
        meet.tile = static_cast<uint32_t>(tile);
        meet.qd = (sub & 1) + 2 * (oy >> 3);           // the 8x8 block of the tile this 8x4 block is half of
        meet.half = (oy >> 2) & 1;
        meet.v = mv;
        meet.open = true;
        const uint32_t wb = __reduce_add_sync(FULL, nb);
        if (lane == 0) {
            if (wb) atomicAdd(J.n_blended, static_cast<unsigned long long>(wb));
            if constexpr (PX == 1)
                meet.old = atomicOr(reinterpret_cast<unsigned long long *>(J.qdone) + 4 * tile + meet.qd,
                                    static_cast<unsigned long long>(meet.prefix + 1u) << (32u * meet.half));
            else
                meet.old = 1ull << (32u * (meet.half ^ 1u));     // an 8x8 block of its own
        }
        if constexpr (PX == 2) meet.settle(batch, lane);
        if (!ahead) take_next(q, nv);
    }
    cp_async_wait<0>();                                 // (what the last item had staged beyond its stop)
    meet.settle(batch, lane);
}

// Backward set-up: the work items (tile, 8x8 block q, segment s) were written
// by the forward as it finished each 8x8 block; this kernel restarts the work
// queue and zeroes the record-gradient rows of the visible Gaussians (visible
// list of the last render, n_vis entries), the only rows the compositor adds
// to and the chain rule reads.
// A thread per 16 bytes, so that consecutive lanes store consecutive words of
// a 48-byte row: 540,000 rows 0.014 ms (a thread per row and 1,024-thread CTAs 0.017).
__global__ void __launch_bounds__(256) k_bwd_setup(uint32_t *__restrict__ queue,
                                                   const uint32_t *__restrict__ vis_index,
                                                   const uint32_t *__restrict__ n_vis, int n,
                                                   float4 *__restrict__ rec_grad) {
    chain_start();
    if (blockIdx.x == 0 && threadIdx.x == 0) *queue = 0;
    const uint64_t words = 3ull * min(*n_vis, static_cast<uint32_t>(n));
    const uint64_t step = static_cast<uint64_t>(gridDim.x) * 256u;
#pragma unroll 4
    for (uint64_t e = blockIdx.x * 256u + threadIdx.x; e < words; e += step) {
        const uint32_t p = static_cast<uint32_t>(e / 3);
        rec_grad[3 * static_cast<size_t>(vis_index[p]) + (e - 3ull * p)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Reduce-scatter of a splat's 10 sums over the 32 lanes in 12 shuffles; lane l
// ends with the warp sum of value reduce10_owner(l).  The four colour values
// are products of one factor with per-lane constants, so each lane forms them
// in the order in which it keeps and sends them (col[0] kept; the sign of the
// lane bit flips the order) and their two halvings need no selects; value 3 or
// 5 stays whole in its half of the warp until the other values have been
// halved away.
__device__ __forceinline__ int reduce10_owner(int lane) {
    const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1, b1 = (lane >> 1) & 1;
    return b1 ? (b4 ? 5 : 3) : (b2 ? (b3 ? (b4 ? 4 : 2) : b4) : 6 + 2 * b4 + b3);
}

// One lane per value: 0, 4, .., 28 and, for values 3 and 5, lanes 2 and 18.
__device__ __forceinline__ bool reduce10_writer(int lane) { return !(lane & 1) && (!(lane & 2) || !(lane & 12)); }

// Which of the colour values 6 .. 9 a lane's slot s holds (less 6).
__device__ __forceinline__ int reduce10_slot(int lane, int s) {
    return 2 * (((lane >> 4) & 1) ^ (s >> 1)) + (((lane >> 3) & 1) ^ (s & 1));
}

// g: values 0 .. 5; col: the colour values in slot order.
__device__ __forceinline__ float reduce_scatter10(const float g[6], const float col[4], int lane) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    const float c0 = col[0] + __shfl_xor_sync(FULL, col[2], 16);
    const float c1 = col[1] + __shfl_xor_sync(FULL, col[3], 16);
    const float p = (b4 ? g[1] : g[0]) + __shfl_xor_sync(FULL, b4 ? g[0] : g[1], 16);
    const float q = (b4 ? g[4] : g[2]) + __shfl_xor_sync(FULL, b4 ? g[2] : g[4], 16);
    float m = (b4 ? g[5] : g[3]) + __shfl_xor_sync(FULL, b4 ? g[3] : g[5], 16);
    const float c = c0 + __shfl_xor_sync(FULL, c1, 8);
    const float x = (b3 ? q : p) + __shfl_xor_sync(FULL, b3 ? p : q, 8);
    m += __shfl_xor_sync(FULL, m, 8);
    const float y = (b2 ? x : c) + __shfl_xor_sync(FULL, b2 ? c : x, 4);
    m += __shfl_xor_sync(FULL, m, 4);
    const float z = (b1 ? m : y) + __shfl_xor_sync(FULL, b1 ? y : m, 2);
    return z + __shfl_xor_sync(FULL, z, 1);
}

// Backward, back to front within a segment.  With
//   S_i = sum_{j>i} c_j a_j T_j + T_N bg   (T_j: transmittance before splat j)
//   dL/da_i = T_i (dC.c_i) - (dC.S_i - dA T_N) / (1 - a_i).
// The scalar R_i = dC.S_i - dA T_N is carried from the back: a work item
// covers list positions [s kSeg, (s+1) kSeg) of one 8x8 block (two pixels per
// lane) and starts from the forward's checkpoint of segment s+1, which holds
// the transmittance there and the colour blended from there on (or from T_N
// and zero when the pixel stopped inside segment s).  Going back, T_i =
// T_{i+1} / (1 - a_i) and R_{i-1} = R_i + (dC.c_i) a_i T_i: every term of R
// is at most of the size of T there, so deep splats keep their relative
// accuracy (a running total minus a prefix would not).
//
// Each splat's 10 sums are reduce-scattered over the warp and added to the
// record gradient, float 12 g + i for value i, by ten lanes at once: with e'
// the natural exponent, E = dL/de', p and dy as in splat_alpha
//   (sum E p, sum E dy, sum E p^2, sum E p dy, sum E dy^2, dopacity, dr, dg, db, sum of alpha*T);
//   contrib_max[g] = max(.., alpha*T).
// The chain rule turns the first five into the gradients of the record's
// geometry (they are linear in them, with factors of the splat alone).
// 1 / (1 - a_i) is the hardware reciprocal approximation (about 1 ulp, exact
// at 1): a correctly rounded reciprocal costs several instructions per pixel
// and splat and changes the gradients only at the last bits.
//
// Bound by instruction issue.  A lane's two pixels go through packed
// arithmetic without branches: a pixel that the splat does not touch takes
// part with alpha 0, and with zeros selected where a product with an infinite
// or undefined value of its own must not count.  Kept splats are staged in
// shared memory with every factor doubled, as the packed instructions want
// them.  1.2M-Gaussian 1024 x 1024 frame 0.198 -> 0.173 ms, 500,000-Gaussian
// 800 x 800 training view 0.148 -> 0.129 (before: one pixel after the other
// behind branches, 220 instructions per splat and block against 160, and the
// geometry's factors applied per splat and block).  The two pixels' products
// are added with one rounding (dot2) and dL/da as a fused difference: packed
// products summed afterwards took 0.166 ms but put twice the rounding noise
// into the quaternion gradients of needle-like splats.  Five CTAs per SM; six
// and seven: 1.2% slower.
struct alignas(16) BwdSplat {
    float2 nax, nay;               // minus the centre
    float2 beta, A2, G2, o;
    float2 r, g;
    float2 b;
    uint32_t gt, pos;              // id with bit 31: trainable; position in the tile's list
};

__global__ void __launch_bounds__(kBwdThreads, 5) k_composite_bwd(
    const uint2 *__restrict__ items, const uint32_t *__restrict__ n_items, uint32_t *__restrict__ queue,
    const uint2 *__restrict__ ranges, const uint32_t *__restrict__ list, const Geo *__restrict__ geo,
    const Rec *__restrict__ rec, int W, int H, int Tx, float3 bg, const float *__restrict__ t_final,
    const uint32_t *__restrict__ n_contrib, const uint32_t *__restrict__ seg_base, const float4 *__restrict__ ckpt,
    const uint32_t *__restrict__ qwork, const float *__restrict__ dL_dimage, const float *__restrict__ dL_dalpha,
    const uint8_t *__restrict__ layer, uint32_t grad_layer_mask, float4 *__restrict__ rec_grad,
    float *__restrict__ contrib_max, uint32_t n_rec, const Ctl *__restrict__ ctl) {
    chain_start();
    __shared__ BwdSplat s_splat[kBwdThreads / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int own = reduce10_owner(lane);
    const bool writer = reduce10_writer(lane);
    const uint32_t total = *n_items;
    const size_t plane = static_cast<size_t>(W) * H;
    for (;;) {
        uint32_t id = 0;
        if (lane == 0) id = atomicAdd(queue, 1u);
        id = __shfl_sync(FULL, id, 0);
        if (id >= total) break;
        const uint2 it = items[total - 1 - id];       // the forward appended the heaviest tiles' items last
        const int tile = static_cast<int>(it.x);
        const int q = static_cast<int>(it.y >> 24);
        const uint32_t seg = it.y & 0xFFFFFFu;
        const uint2 rg = ranges[tile];
        const uint32_t s0 = rg.x + seg * kSeg;
        const int ox = (q & 1) * 8, oy = (q >> 1) * 8;          // the item's 8x8 block of the tile
        const uint32_t s1 = rg.x + min(min((seg + 1) * kSeg, qwork[4 * tile + q]), rg.y - rg.x);
        const float4 *nck = ckpt + (static_cast<size_t>(seg_base[tile]) + seg + 1) * kTilePix;
        const float bx0 = (tile % Tx) * kTile + ox + 0.5f, by0 = (tile / Tx) * kTile + oy + 0.5f;
        // the lane's pixels: rows lane / 8 and lane / 8 + 4 of the block
        float dC[3][2], R[2], T[2];
        uint32_t nc[2];
        const int lx = ox + (lane & 7);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int ly = oy + (lane >> 3) + 4 * j;
            const int x = (tile % Tx) * kTile + lx, y = (tile / Tx) * kTile + ly;
            nc[j] = 0;
            dC[0][j] = dC[1][j] = dC[2][j] = R[j] = 0.f;
            T[j] = 1.f;
            if (x < W && y < H) {
                const size_t pix = static_cast<size_t>(y) * W + x;
                const uint32_t n = n_contrib[pix];
                if (n > seg * kSeg) {
                    nc[j] = n;
                    const float TN = t_final[pix];
                    float dA = 0.f;
                    if (dL_dimage) {
                        dC[0][j] = dL_dimage[pix];
                        dC[1][j] = dL_dimage[plane + pix];
                        dC[2][j] = dL_dimage[2 * plane + pix];
                    }
                    if (dL_dalpha) dA = dL_dalpha[pix];
                    R[j] = TN * (dC[0][j] * bg.x + dC[1][j] * bg.y + dC[2][j] * bg.z) - dA * TN;
                    T[j] = TN;
                    if (n > (seg + 1) * kSeg) {
                        const float4 ck = nck[ly * kTile + lx];
                        T[j] = ck.x;
                        R[j] += dC[0][j] * ck.y + dC[1][j] * ck.z + dC[2][j] * ck.w;
                    }
                }
            }
        }
        // an upstream gradient that is not finite counts for the splats of its own pixel only
        const bool finite = __all_sync(FULL, isfinite(dC[0][0] + dC[0][1]) && isfinite(dC[1][0] + dC[1][1]) &&
                                                 isfinite(dC[2][0] + dC[2][1]));
        const float lpx = (tile % Tx) * kTile + lx + 0.5f, lpy = (tile / Tx) * kTile + oy + (lane >> 3) + 0.5f;
        const F2 px(lpx, lpx), py(lpy, lpy + 4.f);
        const F2 dC0(dC[0][0], dC[0][1]), dC1(dC[1][0], dC[1][1]), dC2(dC[2][0], dC[2][1]);
        F2 kc[4];                   // the colour values' constants in slot order (value 9's is 1)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int v = reduce10_slot(lane, s);
            kc[s] = v == 0 ? dC0 : (v == 1 ? dC1 : (v == 2 ? dC2 : F2(1.f, 1.f)));
        }
        F2 R2(R[0], R[1]), T2(T[0], T[1]);
        const uint32_t nchunk = (s1 - s0 + 31) / 32;
        Chunk nxt;
        // ids one chunk ahead of the splats (the walk goes back to front; every chunk below the last is full)
        uint32_t gid = 0;
        if (nchunk) {
            const uint32_t pos = s0 + (nchunk - 1) * 32 + lane;
            fetch_splat(geo, rec, layer, pos < s1 ? list[pos] : 0u, pos < s1, nxt, n_rec, ctl);
            if (nchunk >= 2) gid = list[pos - 32];
        }
        for (uint32_t c = nchunk; c-- > 0;) {
            const uint32_t base = s0 + c * 32;
            const bool keep = base + lane < s1 && splat_reaches_block(nxt.a, nxt.b, bx0, bx0 + 7.f, by0, by0 + 7.f);
            const unsigned km = __ballot_sync(FULL, keep);
            __syncwarp();
            if (keep) {
                BwdSplat &S = s_splat[warp][__popc(km & lt)];
                const float4 a = nxt.a, b = nxt.b;
                S.nax = make_float2(-a.x, -a.x);
                S.nay = make_float2(-a.y, -a.y);
                S.beta = make_float2(a.w, a.w);
                S.A2 = make_float2(a.z, a.z);
                S.G2 = make_float2(b.x, b.x);
                S.o = make_float2(b.y, b.y);
                S.r = make_float2(b.z, b.z);
                S.g = make_float2(b.w, b.w);
                S.b = make_float2(nxt.c, nxt.c);
                S.gt = nxt.g | (((grad_layer_mask >> nxt.ly) & 1u) << 31);
                S.pos = base + lane - rg.x;
            }
            __syncwarp();
            fetch_splat(geo, rec, layer, gid, c > 0, nxt, n_rec, ctl);
            if (c > 1) gid = list[base - 64 + lane];
            const int cnt = __popc(km);
            for (int k = cnt - 1; k >= 0; --k) {
                const ulonglong2 *S = reinterpret_cast<const ulonglong2 *>(&s_splat[warp][k]);
                const ulonglong2 u0 = S[0], u1 = S[1], u2 = S[2];
                const uint4 u4 = reinterpret_cast<const uint4 *>(S)[4];
                // alpha of both pixels, bit for bit as splat_alpha's
                const F2 dx = add2(px, F2(u0.x)), dy = add2(py, F2(u0.y));
                const F2 p = fma2(F2(u1.x), dy, dx);
                const float2 e = fma2(mul2(F2(u1.y), p), p, mul2(mul2(F2(u2.x), dy), dy)).get();
                const F2 ex(ex2_approx(e.x), ex2_approx(e.y));
                const float2 ao = mul2(F2(u2.y), ex).get();
                const float al0 = fminf(kAlphaMax, ao.x), al1 = fminf(kAlphaMax, ao.y);
                const bool act0 = u4.w < nc[0] && al0 >= kAlphaMin, act1 = u4.w < nc[1] && al1 >= kAlphaMin;
                if (!__any_sync(FULL, act0 || act1)) continue;
                const ulonglong2 u3 = S[3];
                const float a0 = act0 ? al0 : 0.f, a1 = act1 ? al1 : 0.f;
                const F2 al(a0, a1);
                const F2 inv(rcp_approx(__fsub_rn(1.f, a0)), rcp_approx(__fsub_rn(1.f, a1)));
                T2 = mul2(T2, inv);
                const F2 w = mul2(al, T2);
                const float cb = __uint_as_float(u4.x);
                const float2 d = fma2(dC2, F2(cb, cb), fma2(dC1, F2(u3.y), mul2(dC0, F2(u3.x)))).get();
                const F2 dcc(act0 ? d.x : 0.f, act1 ? d.y : 0.f);
                const float2 Rv = R2.get(), iv = inv.get(), t = T2.get(), dc = dcc.get();
                R2 = fma2(w, dcc, R2);
                // dL/da, zero where the product with the opacity was clamped
                const F2 dLda(act0 && ao.x < kAlphaMax ? fmaf(-Rv.x, iv.x, t.x * dc.x) : 0.f,
                              act1 && ao.y < kAlphaMax ? fmaf(-Rv.y, iv.y, t.y * dc.y) : 0.f);
                const F2 E = mul2(dLda, al);
                const F2 tp = mul2(E, p), td = mul2(E, dy);
                const float g[6] = {tp.sum(),     td.sum(),     dot2(tp, p),
                                    dot2(tp, dy), dot2(td, dy), dot2(dLda, ex)};
                float col[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) col[s] = dot2(w, kc[s]);
                const float2 wv = w.get();
                if (!finite) {
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const float2 v = kc[s].get();
                        col[s] = (act0 ? wv.x * v.x : 0.f) + (act1 ? wv.y * v.y : 0.f);
                    }
                }
                const float sv = reduce_scatter10(g, col, lane);
                const uint32_t smx = __reduce_max_sync(FULL, __float_as_uint(fmaxf(wv.x, wv.y)));
                const uint32_t gi = u4.z & 0x7FFFFFFFu;
                // value i is float 12 g + i of the record gradient: one atomic per value, one instruction
                if (writer && ((u4.z >> 31) || own == 9))
                    atomicAdd(reinterpret_cast<float *>(rec_grad) + 12 * static_cast<size_t>(gi) + own, sv);
                if (lane == 1 && contrib_max) atomicMax(reinterpret_cast<unsigned int *>(&contrib_max[gi]), smx);
            }
        }
    }
}

// Blocks that fill every SM once for a persistent kernel.
template <class K>
int persistent_blocks(K kernel, int threads, size_t smem = 0) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (smem) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
    return max(1, sms) * max(1, per);
}

// Pixels of a launch from which the forward takes two pixels per lane.  Below,
// the few longest walks set the time and an 8x8 block's walk is longer than an
// 8x4 block's (1024x1024 frame 0.126 against 0.114 ms, 1037x771 view 0.137 against
// 0.096); above, the work per pixel does (1920x1080 view 0.211 against 0.316 ms,
// 2064x2208 view 0.452 against 0.697, eight 512x512 views in one launch 0.274
// against 0.280).
constexpr uint64_t kFwdWidePixels = 3u << 19;

// One launch of the forward compositor: every SM filled once.
template <int PX, int PER>
cudaError_t launch_forward(const FwdBatch &batch, uint32_t items, cudaStream_t st) {
    constexpr size_t smem = sizeof(FwdSmem<PER>);
    static PerDevice cache;
    const int blocks = cache.get([] { return persistent_blocks(k_composite_fwd<PX, PER>, kFwdThreads, smem); });
    const uint32_t need = (items + kFwdWarps - 1) / kFwdWarps;
    launch_chained(k_composite_fwd<PX, PER>, min(static_cast<uint32_t>(blocks), need), kFwdThreads, smem, st, batch);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_composite_forward(const FwdJob *jobs, int n, cudaStream_t st) {
    FwdBatch batch;
    batch.n = 0;
    uint32_t total = 0;
    uint64_t pixels = 0;
    for (int i = 0; i < n && batch.n < kMaxBatch; ++i) {
        if (jobs[i].Tn == 0) continue;
        batch.job[batch.n++] = jobs[i];
        total += static_cast<uint32_t>(jobs[i].Tn) * 8u;
        pixels += static_cast<uint64_t>(jobs[i].W) * jobs[i].H;
    }
    if (total == 0) return cudaSuccess;
    return pixels >= kFwdWidePixels ? launch_forward<2, 2>(batch, total / 2, st)
                                    : launch_forward<1, 4>(batch, total, st);
}

cudaError_t launch_bwd_setup(const CompositeBufs &cb, int Tx, int Ty, float4 *rec_grad, const uint32_t *vis_index,
                             const uint32_t *n_vis, int n, cudaStream_t st) {
    if (Tx * Ty == 0) return cudaSuccess;
    static PerDevice cache;
    const int sms = cache.get([] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return max(1, v);
    });
    const int64_t want = (3ll * n + 1023) / 1024;                // four words a thread, at most eight CTAs per SM
    const int blocks = static_cast<int>(want < 8ll * sms ? (want > 1 ? want : 1) : 8ll * sms);
    k_bwd_setup<<<blocks, 256, 0, st>>>(cb.queue, vis_index, n_vis, n, rec_grad);
    return cudaGetLastError();
}

cudaError_t launch_composite_backward(const CompositeBufs &cb, const uint2 *ranges, const uint32_t *list,
                                      const Geo *geo, const Rec *rec, int W, int H, int Tx, int Ty, float3 bg,
                                      const float *t_final, const uint32_t *n_contrib, const float *dL_dimage,
                                      const float *dL_dalpha, const uint8_t *layer, uint32_t grad_layer_mask,
                                      float4 *rec_grad, float *contrib_max, uint32_t n, const Ctl *ctl,
                                      cudaStream_t st) {
    if (Tx * Ty == 0) return cudaSuccess;
    static PerDevice cache;
    const int blocks = cache.get([] { return persistent_blocks(k_composite_bwd, kBwdThreads); });
    launch_chained(k_composite_bwd, blocks, kBwdThreads, 0, st, cb.items, cb.n_items, cb.queue, ranges, list, geo,
                   rec, W, H, Tx, bg, t_final, n_contrib, cb.seg_base, cb.ckpt, cb.qwork, dL_dimage, dL_dalpha, layer,
                   grad_layer_mask, rec_grad, contrib_max, n, ctl);
    return cudaGetLastError();
}

}  // namespace gs
