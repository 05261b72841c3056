// SH codebook (Sec. 3.3: the SH coefficients, about 3/4 of a model's size,
// are clustered with K-means across all layers; Sec. 4.3).  Lloyd's
// iteration on the device, then encoding: every Gaussian keeps its DC
// coefficient and stores a 16-bit index into an FP16 table of the remaining
// 3(K-1) coefficients.  The preprocess gathers those rows from L2 instead of
// reading 3(K-1) floats per Gaussian from HBM.
//
// Assignment: the centroid with the least single-precision distance
// sum_d (x_d - c_d)^2 (d in order, fused multiply-adds), ties to the lower
// index.  Small calls scan brute force: a thread per point holds its
// (zero-padded) coordinates in registers and scans the centroids staged in
// shared memory 64 at a time with 16-byte broadcast loads (scan_all).  Larger
// ones rule out nearly all centroids on the tensor cores first
// (k_kmeans_assign_tc).
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kKmTile = 64;                  // centroids per shared-memory tile
constexpr int kKmThreads = 128;

// The brute-force scan of point i by one thread of a CTA of NT (i >= n: none), over D >= dim coordinates (the others
// are zero).  Two centroids go through packed arithmetic together, each in the order of its coordinates, and two such
// pairs are in flight: with a warp per scheduler the loop waits on the chains, with more it is bound by 2 D operations
// per point and centroid.  Centroids are staged negated and interleaved in pairs; those past the end are infinitely
// far.  One centroid at a time over 48 coordinates, before: 512 points x 16,384 centroids of 45 coordinates 2.99 -> 1.93
// ms, 20,000 x 127 0.038 -> 0.032, 1,000,000 x 100 of 24 coordinates 0.393 -> 0.197, 1,000 x 64 of 9 0.020 -> 0.012.
struct ScanTile {
    float4 c[kKmTile / 2][kCbMaxDim / 2];
};
template <int NT, int D>
__device__ __forceinline__ uint32_t scan_all(const float *__restrict__ pts, int64_t i, int64_t n, int dim,
                                             int64_t stride, const float *__restrict__ cent, int k, ScanTile &s) {
    // x doubled for the packed operations; `zero` (k is positive, which the compiler does not know) keeps both halves in
    // registers, where they would else be put together by moves before every use (20,000 x 2,048 0.42 against 0.33 ms)
    const uint32_t zero = static_cast<uint32_t>(k) >> 31;
    F2 x[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const float v = (i < n && d < dim) ? pts[i * stride + d] : 0.f;
        x[d] = F2(v, __uint_as_float(__float_as_uint(v) ^ zero));
    }
    float best = 3.0e38f;
    uint32_t arg = 0;
    for (int t0 = 0; t0 < k; t0 += kKmTile) {
        __syncthreads();
        for (int e = threadIdx.x; e < kKmTile * D; e += NT) {
            const int j = e / D, d = e % D;
            const float v = t0 + j >= k ? INFINITY : (d < dim ? cent[(t0 + j) * dim + d] : 0.f);
            reinterpret_cast<float *>(&s.c[j >> 1][0])[2 * d + (j & 1)] = -v;
        }
        __syncthreads();
        const int m = min(kKmTile, k - t0);
        for (int j = 0; j < m; j += 4) {
            F2 acc[2] = {F2(0.f, 0.f), F2(0.f, 0.f)};
#pragma unroll
            for (int q = 0; q < D / 2; ++q) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float4 c = s.c[j / 2 + u][q];
                    const F2 a = add2(x[2 * q], F2(c.x, c.y)), b = add2(x[2 * q + 1], F2(c.z, c.w));
                    acc[u] = fma2(b, b, fma2(a, a, acc[u]));
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float2 r = acc[u].get();
                if (r.x < best) {
                    best = r.x;
                    arg = static_cast<uint32_t>(t0 + j + 2 * u);
                }
                if (r.y < best) {
                    best = r.y;
                    arg = static_cast<uint32_t>(t0 + j + 2 * u + 1);
                }
            }
        }
    }
    return arg;
}

template <int D>
__global__ void __launch_bounds__(kKmThreads) k_kmeans_assign(const float *__restrict__ pts, int64_t n, int dim,
                                                              int64_t stride, const float *__restrict__ cent, int k,
                                                              uint32_t *__restrict__ assign) {
    __shared__ ScanTile s_c;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kKmThreads + threadIdx.x;
    const uint32_t arg = scan_all<kKmThreads, D>(pts, i, n, dim, stride, cent, k, s_c);
    if (i < n) assign[i] = arg;
}

// ---- assignment on the tensor cores ----
//
// argmin_c |x - c|^2 = argmax_c s(c), s(c) = x.c - |c|^2 / 2: a contraction of
// the points with the centroids.  The kernel computes s in bf16 products with
// FP32 accumulation (tcgen05), bounds its error, and evaluates the exact
// single-precision distance only for the centroids that the bounds leave, so
// the result is that of the brute-force scan, bit for bit:
//
//  * |s~(c) - s(c)| <= E = |x||c| (2^-8 + 2^-18 + 2^-16) + |c|^2 2^-16: both
//    factors of a product are rounded to 8 bits (relative 2^-9 each;
//    Cauchy-Schwarz over the coordinates), -|c|^2/2 enters as three bf16
//    parts, and each of at most 64 accumulations errs by at most 2^-22 of the
//    magnitudes added.  kEProd, kENorm round these up; kETiny covers underflow.
//    (The last of the three is an assumption: the rounding of the accumulation is
//    not documented.  The constants leave room for 2^-20.)
//  * The scan's rounded distances err by at most (dim + 3) 2^-24 relative, so
//    its winner has s within 2^-18 (|x| + |c|)^2 of the best; kESlack rounds up.
//  * Per point, LB = max over groups of 32 centroids of (largest s~ - E) is a lower
//    bound of the best s.  A centroid whose s~ + E + slack stays below LB cannot be
//    the winner.  The others are remembered (with U, that sum for the group's
//    largest; kCand at most, dropped again when LB has passed them).
//  * Points whose candidates overflow, and points and centroids that are not
//    finite or above kHuge, are scanned in full.
//
// A CTA takes 256 points (two 128-row A tiles, bf16, resident) and walks the
// centroids in tiles of 128: two sets of four warps take the tiles in turn, each
// tile's rows by one bulk copy, and convert them to bf16 in the 128-byte swizzled
// K-major layout, one thread issues the MMAs (M = N = 128, K = dim + 3 rounded up
// to 16) into one of two accumulator sets in tensor memory, and eight warps read
// the other set back, one point per thread.  Everything is staged by the CTA
// itself, as the entry point has no workspace to hold converted centroids.
//
// Bound by the latencies of that chain: half of the issue slots are used, the
// tensor pipe is 19% busy (K is only 48), and what is waited for are the tile
// hand-overs and the accumulators.  Measured, points x centroids of 45
// coordinates against the scan of one centroid at a time: 200,000 x 16,384 13.0 -> 0.81
// ms, 200,000 x 4,096 3.26 -> 0.32, 1,200,000 x 16,384 71.9 -> 4.2, 20,000 x 256 0.064 ->
// 0.031; 20,000 x 16,384 of 9 coordinates 3.3 -> 0.13.  Found on the way: candidate groups
// scanned whole by a warp per point (1.1 ms: a kilobyte-sized gather per point), one
// converter set (1.2 ms), candidates told apart by 32 predicates (1.0 ms, the sign
// bits 0.79).  Data of few colours leave many candidates: see k_kmeans_assign_left.
constexpr int kTcPoints = 256, kTcTile = 128, kTcRow = 128;      // points per CTA, centroids per tile, bytes per row
constexpr int kTcEpiWarps = 8, kTcCvtWarps = 4, kTcCvtSets = 2;
constexpr int kTcMmaWarp = kTcEpiWarps + kTcCvtSets * kTcCvtWarps;
constexpr int kTcThreads = 32 * (kTcMmaWarp + 1);
constexpr int kCand = 16;              // candidate groups remembered per point
// A point with more than this share of the centroids left is scanned in full.  Evaluated one by one, 200,000 points with
// 128 of 512 centroids left took 0.87 ms, with 64 0.53, with 32 0.40; with the scan 0.55, 0.52 and 0.69 (half of the
// points, but every CTA).
constexpr int kCandShare = 6;
constexpr int kCmRing = 8;             // tiles whose largest norms are kept
constexpr float kEProd = 1.05f * 0x1p-8f, kENorm = 0x1p-15f, kESlack = 0x1p-17f, kETiny = 1e-30f, kHuge = 1e14f;
constexpr uint32_t kTcWaitLimit = 1u << 22;
#ifdef GS_DEBUG
__device__ uint32_t g_dbg_tc_wait = kTcWaitLimit;      // test hook (gs_debug_kmeans_wait)
#endif
constexpr uint32_t kUnassigned = 0xFFFFFFFFu;
// Calls from this size on go through the tensor cores (20,000 points: 128 centroids
// 0.025 ms against 0.033 for the scan, 64 centroids 0.019 with the scan; 1,024 points
// x 128 centroids 0.023 against 0.029).
constexpr int kTcMinCentroids = 128;
constexpr int64_t kTcMinPoints = 1024;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// The scan's distance, accumulated in the order of the coordinates.
__device__ __forceinline__ float sq_step(float x, float c, float acc) {
    const float a = __fsub_rn(x, c);
    return __fmaf_rn(a, a, acc);
}

// A point and the rows of a group of 32 centroids in shared memory, by cp.async.
struct __align__(16) PairBuf {
    float rows[32 * kCbMaxDim];
    float x[kCbMaxDim];
    uint32_t g;

    // vec: cent is 16-byte aligned (so is every group: 32 rows are a multiple of 128 bytes).
    __device__ __forceinline__ void fetch(const float *__restrict__ cent, int k, int dim, uint32_t group,
                                          const float *__restrict__ pt, bool vec, int lane) {
        const int vals = min(32, k - static_cast<int>(32u * group)) * dim;
        const float *src = cent + static_cast<size_t>(32u * group) * dim;
        const uint32_t dst = smem_u32(rows);
        const int units = vec ? vals / 4 : 0;
#pragma unroll
        for (int j = 0; j < 32 * kCbMaxDim / 128; ++j) {
            const int u = lane + 32 * j;
            if (u < units)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * u), "l"(src + 4 * u)
                             : "memory");
        }
        for (int v = 4 * units + lane; v < vals; v += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * v), "l"(src + v) : "memory");
        for (int d = lane; d < dim; d += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(x + d)), "l"(pt + d) : "memory");
        if (lane == 0) g = group;
    }
    // The least distance of the point to the group, a centroid per lane; keeps (best, arg) the scan's winner so far
    // when groups come in ascending order.
    __device__ __forceinline__ void least(int k, int dim, int lane, float &best, uint32_t &arg) const {
        const bool row = static_cast<int>(32u * g) + lane < k;
        const float *c = rows + (row ? lane : 0) * dim;
        float acc = 0.f;
#pragma unroll
        for (int d = 0; d < kCbMaxDim; ++d)
            if (d < dim) acc = sq_step(x[d], c[d], acc);
        const bool in = row && acc < best;
        const uint32_t bits = in ? __float_as_uint(acc) : 0xFFFFFFFFu;       // distances are not negative
        const uint32_t low = __reduce_min_sync(0xFFFFFFFFu, bits);
        if (low != 0xFFFFFFFFu) {
            best = __uint_as_float(low);
            arg = 32u * g + static_cast<uint32_t>(__ffs(__ballot_sync(0xFFFFFFFFu, bits == low)) - 1);
        }
    }
};

struct TcOperands {
    unsigned char a[2][128 * kTcRow];              // points, bf16 (1024-byte aligned)
    unsigned char b[2][kTcTile * kTcRow];          // centroid tiles, bf16
    float rows[2][kTcTile * kCbMaxDim];            // centroid rows as they are in memory
};
struct TcSmem {
    TcOperands op;
    float2 cand[kCand][kTcPoints];                 // (U, group of 32 centroids)
    uint32_t mask[kCand][kTcPoints];               // the group's centroids that can still win
    float4 cm[kCmRing];                            // largest |c| of a tile, per converting warp
    unsigned long long row_full[kTcCvtSets], b_full[2], b_empty[2], acc_full[2], acc_empty[2];
    uint32_t tmem;
    int failed, quit[kTcCvtSets];
};

__device__ __forceinline__ void mbar_init(void *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(void *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Waits for the phase of the given parity; false when the limit runs out or another role has given up (`failed`; with
// null the wait is for work of this thread's own that is under way, whatever the others do).
__device__ __forceinline__ bool mbar_wait(void *bar, uint32_t parity, volatile int *failed) {
    const uint32_t addr = smem_u32(bar);
#ifdef GS_DEBUG
    const uint32_t limit = failed ? g_dbg_tc_wait : kTcWaitLimit;
#else
    constexpr uint32_t limit = kTcWaitLimit;
#endif
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (ok) return true;
        if (failed && *failed) return false;
    }
    if (failed) *failed = 1;
    return false;
}

// Shared-memory matrix descriptor: K-major rows of 128 bytes, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr) {
    return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// kind::f16: D f32, A and B bf16, both K-major, M = N = 128.
constexpr uint32_t kUmmaInstr = (1u << 4) | (1u << 7) | (1u << 10) | ((kTcTile / 8u) << 17) | ((128u / 16u) << 24);

__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(kUmmaInstr), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(void *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 consecutive accumulator columns of the warp's 32 rows, a row per lane; v is valid after tmem_wait(v), which also
// waits for every other load of the warp.
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {"
        "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31"
        "}, [%32];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
          "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
          "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
        : "r"(addr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait(float (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
        : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
          "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]),
          "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]),
          "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]), "+f"(v[30]), "+f"(v[31])
        :
        : "memory");
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float m;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
    return m;
}

// Byte offset of 16-byte unit u of row r in the 128-byte swizzled layout.
__device__ __forceinline__ uint32_t swz(uint32_t r, uint32_t u) { return r * kTcRow + ((u ^ (r & 7u)) << 4); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// DIM: the coordinates where known at compile time (SH degrees 1 to 3), 0 otherwise.
template <int DIM>
__global__ void __launch_bounds__(kTcThreads) k_kmeans_assign_tc(const float *__restrict__ pts, int64_t n, int dim_,
                                                                 int64_t stride, const float *__restrict__ cent, int k,
                                                                 uint32_t *__restrict__ assign) {
    const int dim = DIM ? DIM : dim_;
    extern __shared__ unsigned char s_raw[];
    TcSmem &sm = *reinterpret_cast<TcSmem *>((reinterpret_cast<uintptr_t>(s_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kTcPoints;
    const int ntile = (k + kTcTile - 1) / kTcTile;
    const int ksteps = (dim + 3 + 15) / 16;
    volatile int *failed = &sm.failed;
    if (threadIdx.x == 0) {
        sm.failed = sm.quit[0] = sm.quit[1] = 0;
        for (int q = 0; q < 2; ++q) {
            mbar_init(&sm.b_full[q], 32 * kTcCvtWarps);
            mbar_init(&sm.b_empty[q], 1);
            mbar_init(&sm.row_full[q], 1);
            mbar_init(&sm.acc_full[q], 1);
            mbar_init(&sm.acc_empty[q], 32 * kTcEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kTcMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm.tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the points: bf16 rows (x, 1, 1, 1, 0 ...), 32 rows per warp, two coordinates per lane
    float nx = 0.f;                                            // |x| of point `threadIdx.x` (rounded up)
    if (warp < kTcEpiWarps) {
        constexpr int R = 8;                                   // rows whose loads are in flight together
        for (int r0 = 0; r0 < 32; r0 += R) {
            float2 x[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = i0 + 32 * warp + r0 + r;
                x[r] = make_float2(i < n && lane < dim ? pts[i * stride + lane] : 0.f,
                                   i < n && lane + 32 < dim ? pts[i * stride + lane + 32] : 0.f);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float sq = x[r].x * x[r].x + x[r].y * x[r].y;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
                if (lane == r0 + r) nx = sqrtf(sq) * 1.0001f;
                const int row = 32 * warp + r0 + r;
                unsigned char *t = sm.op.a[row >> 7];
                const uint32_t rr = row & 127;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int d = lane + 32 * h;
                    const float v = d < dim ? (h ? x[r].y : x[r].x) : (d < dim + 3 ? 1.f : 0.f);
                    *reinterpret_cast<__nv_bfloat16 *>(t + swz(rr, d >> 3) + 2 * (d & 7)) = __float2bfloat16_rn(v);
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sm.tmem;

    int cnt = 0;                                               // epilogue: candidates of this thread's point
    float LB = -3.0e38f;
    bool full = false;
    if (warp < kTcEpiWarps) {
        full = !(nx < kHuge);
        float cmax = 0.f;
        const int tid = threadIdx.x;
        const uint32_t row = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + (warp >= 4 ? kTcTile : 0);
        for (int t = 0; t < ntile; ++t) {
            const int q = t & 1;
            if (!__all_sync(0xFFFFFFFFu, mbar_wait(&sm.acc_full[q], (t >> 1) & 1, failed))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const float4 c4 = sm.cm[t & (kCmRing - 1)];
            const float cm = fmaxf(fmaxf(c4.x, c4.y), fmaxf(c4.z, c4.w));
            const bool sane = cm < kHuge;                      // (a NaN norm is reported as infinite)
            if (sane) cmax = fmaxf(cmax, cm);
            const float E = nx * cm * kEProd + cm * cm * kENorm + kETiny;
            const float both = nx + cmax;
            const float up = E + both * both * kESlack;
            float v[2][32];                                    // the next group's columns load while one is searched
            tmem_ld32(row + q * 2 * kTcTile, v[0]);
#pragma unroll
            for (int g = 0; g < kTcTile / 32; ++g) {
                float (&w)[32] = v[g & 1];
                tmem_wait(w);
                if (g + 1 < kTcTile / 32) tmem_ld32(row + q * 2 * kTcTile + 32 * (g + 1), v[(g + 1) & 1]);
                do {
                    float m3[10];
#pragma unroll
                    for (int e = 0; e < 10; ++e) m3[e] = max3(w[3 * e], w[3 * e + 1], w[3 * e + 2]);
                    const float m = max3(max3(m3[0], m3[1], m3[2]), max3(m3[3], m3[4], m3[5]),
                                         max3(max3(m3[6], m3[7], m3[8]), m3[9], fmaxf(w[30], w[31])));
                    const int grp = t * (kTcTile / 32) + g;
                    if (32 * grp >= k) break;
                    if (sane) LB = fmaxf(LB, m - E);
                    const float U = sane ? m + up : INFINITY;
                    if (U >= LB && !full) {
                        // the group's centroids that can still win: the sign bits of s~ - (LB - up)
                        const float least = LB - up;
                        uint32_t below = 0;
#pragma unroll
                        for (int e = 31; e >= 0; --e)
                            below = __funnelshift_l(__float_as_uint(w[e] - least), below, 1);
                        if (cnt == kCand) {                    // drop what LB has passed
                            int kept = 0;
                            for (int e = 0; e < kCand; ++e) {
                                const float2 z = sm.cand[e][tid];
                                if (z.x >= LB) {
                                    sm.cand[kept][tid] = z;
                                    sm.mask[kept++][tid] = sm.mask[e][tid];
                                }
                            }
                            cnt = kept;
                        }
                        if (cnt < kCand) {
                            sm.cand[cnt][tid] = make_float2(U, __int_as_float(grp));
                            sm.mask[cnt++][tid] = sane ? ~below : 0xFFFFFFFFu;
                        } else {
                            full = true;
                        }
                    }
                } while (false);
                __syncwarp();
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&sm.acc_empty[q]);
        }
    } else if (warp < kTcMmaWarp) {
        // converters, two sets of four warps taking the tiles in turn: thread r of a set owns centroid row r
        const int set = (warp - kTcEpiWarps) / kTcCvtWarps, cw = (warp - kTcEpiWarps) % kTcCvtWarps;
        const int r = 32 * cw + lane;
        float *const mem = sm.op.rows[set];
        const bool vec = (reinterpret_cast<uintptr_t>(cent) & 15u) == 0;
        const auto set_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "n"(32 * kTcCvtWarps) : "memory"); };
        volatile int *quit = &sm.quit[set];                    // (written before the barrier by thread 0, read behind it)
        bool copying = false;                                  // (thread 0 of the set: a bulk copy is under way)
        // A tile's rows, one bulk copy of whole 16-byte units (a last tile's odd values by plain loads); centroids
        // that do not start on 16 bytes value by value.
        const auto fetch = [&](int t) {
            if (t >= ntile) return;
            const int vals = min(kTcTile, k - t * kTcTile) * dim;
            const float *src = cent + static_cast<size_t>(t) * kTcTile * dim;
            const int bulk = vec ? vals & ~3 : 0;
            if (vec && r == 0 && bulk == 0) mbar_arrive(&sm.row_full[set]);      // (a copy has to have a size)
            if (vec && r == 0 && bulk > 0) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&sm.row_full[set])),
                             "r"(4 * bulk)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        smem_u32(mem)),
                    "l"(src), "r"(4 * bulk), "r"(smem_u32(&sm.row_full[set]))
                    : "memory");
                copying = true;
            }
            for (int e = bulk + r; e < vals; e += 32 * kTcCvtWarps) mem[e] = src[e];
        };
        fetch(set);
        for (int t = set; t < ntile; t += kTcCvtSets) {
            const int q = t & 1;
            // A wait that gives up is noted in `failed`: the CTA's points are then scanned in full.  The set leaves
            // the walk as one, behind its own copy, which must not land in the shared memory of a later CTA.
            const bool landed = !vec || mbar_wait(&sm.row_full[set], (t / kTcCvtSets) & 1, failed);
            if (landed) copying = false;
            if (r == 0 && (!landed || *failed)) *quit = 1;
            set_sync();                                        // the tile's rows have landed
            if (*quit) {
                if (copying) mbar_wait(&sm.row_full[set], (t / kTcCvtSets) & 1, nullptr);
                break;
            }
            const bool in = t * kTcTile + r < k;
            const float *src = mem + r * dim;
            float sq = 0.f;
            uint32_t w[32];                                    // the row's 64 bf16
#pragma unroll
            for (int d = 0; d < kCbMaxDim; d += 2) {
                const float a = in && d < dim ? src[d] : 0.f, b = in && d + 1 < dim ? src[d + 1] : 0.f;
                sq = fmaf(a, a, sq);
                sq = fmaf(b, b, sq);
                w[d / 2] = pack_bf16(a, b);
            }
#pragma unroll
            for (int d = kCbMaxDim / 2; d < 32; ++d) w[d] = 0u;
            // the tile's largest norm; one that is not a number or too large makes its groups candidates
            float nc = sqrtf(sq) * 1.0001f;
            if (!(nc < kHuge)) nc = INFINITY;
            const float wm = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(nc)));
            if (lane == 0) reinterpret_cast<float *>(&sm.cm[t & (kCmRing - 1)])[cw] = wm;
            // The set's next tile goes into the same rows by a bulk copy (async proxy): every thread's reads come
            // before it.  The norm stored above depends on all reads of the warp, and the fence orders the proxies; with
            // the barrier alone a read still in the queue could return the next tile's values.
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            set_sync();
            fetch(t + kTcCvtSets);
            if (t >= 2) mbar_wait(&sm.b_empty[q], ((t >> 1) - 1) & 1, failed);
            // -|c|^2 / 2 in three parts at dim .. dim + 2; a row past the end scores far below any other
            const float h = in ? 0.5f * sq : 1e30f;
            float part[3];
            part[0] = __bfloat162float(__float2bfloat16_rn(h));
            part[1] = __bfloat162float(__float2bfloat16_rn(h - part[0]));
            part[2] = h - part[0] - part[1];
            unsigned char *row = sm.op.b[q];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                *reinterpret_cast<uint4 *>(row + swz(r, u)) =
                    make_uint4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
#pragma unroll
            for (int z = 0; z < 3; ++z)
                *reinterpret_cast<__nv_bfloat16 *>(row + swz(r, (dim + z) >> 3) + 2 * ((dim + z) & 7)) =
                    __float2bfloat16_rn(-part[z]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&sm.b_full[q]);
        }
    } else if (lane == 0) {
        const uint64_t da[2] = {umma_desc(smem_u32(sm.op.a[0])), umma_desc(smem_u32(sm.op.a[1]))};
        const uint64_t db[2] = {umma_desc(smem_u32(sm.op.b[0])), umma_desc(smem_u32(sm.op.b[1]))};
        int t = 0;
        for (; t < ntile; ++t) {
            const int q = t & 1;
            if (!mbar_wait(&sm.b_full[q], (t >> 1) & 1, failed)) break;
            if (t >= 2 && !mbar_wait(&sm.acc_empty[q], ((t >> 1) - 1) & 1, failed)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int m = 0; m < 2; ++m)
                for (int s = 0; s < ksteps; ++s)
                    umma_bf16(tmem + q * 2 * kTcTile + m * kTcTile, da[m] + 2 * s, db[q] + 2 * s, s > 0);
            umma_commit(&sm.b_empty[q]);
            umma_commit(&sm.acc_full[q]);
        }
        // the MMAs that were issued (the last two tiles') have completed before the tensor memory is freed
        for (int u = max(0, t - 2); u < t; ++u) {
            mbar_wait(&sm.b_empty[u & 1], (u >> 1) & 1, nullptr);
            mbar_wait(&sm.acc_full[u & 1], (u >> 1) & 1, nullptr);
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == kTcMmaWarp) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
        return;
    }
    if (warp >= kTcEpiWarps) return;
    // exact distances of the centroids that are left, a point per thread
    const int64_t i = i0 + threadIdx.x;
    if (i >= n) return;
    uint32_t arg = kUnassigned;                                // (scanned in full by the next launch)
    // (32 a group at most: only few centroids can be left in large part)
    const int most = max(8, k / kCandShare);
    int ncand = 0;
    if (32 * cnt > most)
        for (int e = 0; e < cnt; ++e)
            if (sm.cand[e][threadIdx.x].x >= LB) ncand += __popc(sm.mask[e][threadIdx.x]);
    if (!full && !*failed && ncand <= most) {
        const float *pt = pts + i * stride;
        float x[kCbMaxDim];
#pragma unroll
        for (int d = 0; d < kCbMaxDim; ++d) x[d] = d < dim ? pt[d] : 0.f;
        float best = 3.0e38f;
        arg = 0;
        for (int e = 0; e < cnt; ++e) {                        // ascending
            const float2 z = sm.cand[e][threadIdx.x];
            if (!(z.x >= LB)) continue;
            const uint32_t j0 = 32u * static_cast<uint32_t>(__float_as_int(z.y));
            for (uint32_t mask = sm.mask[e][threadIdx.x]; mask; mask &= mask - 1) {
                const uint32_t j = j0 + static_cast<uint32_t>(__ffs(mask) - 1);
                if (j >= static_cast<uint32_t>(k)) break;
                const float *c = cent + static_cast<size_t>(j) * dim;
                float y[kCbMaxDim];
#pragma unroll
                for (int d = 0; d < kCbMaxDim; ++d) y[d] = d < dim ? c[d] : 0.f;
                float acc = 0.f;
#pragma unroll
                for (int d = 0; d < kCbMaxDim; ++d) acc = sq_step(x[d], y[d], acc);
                if (acc < best) {
                    best = acc;
                    arg = j;
                }
            }
        }
    }
    assign[i] = arg;
}

// The points that k_kmeans_assign_tc left (kUnassigned), in full: a CTA per kLeftPoints points collects those left
// among them.  A few are scanned a warp per point, many a thread per point.  Their count comes from the barrier, which
// makes the scan's loops uniform; taken from shared memory, the same loop took 0.75 against 0.47 ms (20,000 points x
// 2,048 centroids).  Colours of a palette are what the bounds leave: 200,000 points of 64 colours x 16,384 centroids
// 15.2 -> 13.0 ms in all (a spread of 0.1 of the palette's; 0.3: 15.7 -> 13.5; all points scanned without the tensor cores
// 13.04), 50,000 x 4,096 of 24 coordinates 1.62 -> 0.64 (1.01), 20,000 x 2,048 0.78 -> 0.38 (0.43).
constexpr int kLeftPoints = 128;

template <int D>
__global__ void __launch_bounds__(kLeftPoints) k_kmeans_assign_left(const float *__restrict__ pts, int64_t n, int dim,
                                                                    int64_t stride, const float *__restrict__ cent,
                                                                    int k, uint32_t *__restrict__ assign) {
    __shared__ __align__(16) union {
        ScanTile c;
        PairBuf pair[kLeftPoints / 32];
    } s;
    __shared__ int s_left[kLeftPoints];
    __shared__ int s_n;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kLeftPoints;
    const bool left = i0 + threadIdx.x < n && assign[i0 + threadIdx.x] == kUnassigned;
    if (threadIdx.x == 0) s_n = 0;
    const int m = __syncthreads_count(left);
    if (m == 0) return;
    if (left) s_left[atomicAdd(&s_n, 1)] = threadIdx.x;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool vec = (reinterpret_cast<uintptr_t>(cent) & 15u) == 0;
    if (m <= kLeftPoints / 8) {
        for (int p = warp; p < m; p += kLeftPoints / 32) {
            const int64_t i = i0 + s_left[p];
            float best = 3.0e38f;
            uint32_t arg = 0;
            for (int g = 0; 32 * g < k; ++g) {
                s.pair[warp].fetch(cent, k, dim, g, pts + i * stride, vec, lane);
                asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
                __syncwarp();
                s.pair[warp].least(k, dim, lane, best, arg);
                __syncwarp();
            }
            if (lane == 0) assign[i] = arg;
        }
        return;
    }
    const int64_t i = static_cast<int>(threadIdx.x) < m ? i0 + s_left[threadIdx.x] : n;
    const uint32_t arg = scan_all<kLeftPoints, D>(pts, i, n, dim, stride, cent, k, s.c);
    if (i < n) assign[i] = arg;
}

// Cluster sums and counts, a warp per point: the lanes hold its coordinates, so
// a row is read and added in whole lines (a thread per point touched a line per
// coordinate and lane), four points in flight.  200,000 points of 45
// coordinates into 16,384 clusters 0.072 -> 0.027 ms (the whole update), into 128
// clusters 0.363 -> 0.094.
__global__ void __launch_bounds__(256) k_kmeans_accumulate(const float *__restrict__ pts, int64_t n, int dim,
                                                           int64_t stride, const uint32_t *__restrict__ assign,
                                                           float *__restrict__ sums, float *__restrict__ cnt) {
    constexpr int P = 4;
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x / 32) + (threadIdx.x >> 5); i < n; i += P * warps) {
        uint32_t a[P];
        float x[P][2];
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const int64_t j = i + q * warps;
            a[q] = j < n ? assign[j] : 0u;
            x[q][0] = j < n && lane < dim ? pts[j * stride + lane] : 0.f;
            x[q][1] = j < n && lane + 32 < dim ? pts[j * stride + lane + 32] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < P; ++q) {
            if (i + q * warps >= n) break;
            float *row = sums + static_cast<size_t>(a[q]) * dim;
            if (lane < dim) atomicAdd(row + lane, x[q][0]);
            if (lane + 32 < dim) atomicAdd(row + lane + 32, x[q][1]);
            if (lane == 31) atomicAdd(&cnt[a[q]], 1.f);
        }
    }
}

__global__ void __launch_bounds__(256) k_kmeans_finish(const float *__restrict__ sums, const float *__restrict__ cnt,
                                                       int k, int dim, float *__restrict__ cent) {
    const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (e >= static_cast<int64_t>(k) * dim) return;
    const float c = cnt[e / dim];
    if (c > 0.f) cent[e] = sums[e] / c;
}

// DC copy, 16-bit indices and the FP16 table (rows padded to `row` halves).
__global__ void __launch_bounds__(256) k_sh_encode(const float *__restrict__ sh, int64_t n, int K,
                                                   const uint32_t *__restrict__ assign, const float *__restrict__ cent,
                                                   int k, int row, float *__restrict__ dc,
                                                   uint16_t *__restrict__ index, __half *__restrict__ table) {
    const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    const int dim = 3 * (K - 1);
    if (e < n) {
        dc[3 * e] = sh[e * 3 * K];
        dc[3 * e + 1] = sh[e * 3 * K + 1];
        dc[3 * e + 2] = sh[e * 3 * K + 2];
        index[e] = static_cast<uint16_t>(assign[e]);
    }
    if (e < static_cast<int64_t>(k) * row) {
        const int64_t j = e / row, d = e % row;
        table[e] = __float2half_rn(d < dim ? cent[j * dim + d] : 0.f);
    }
}

// f(the scanned width as a constant): the least even one for the rows of SH degrees 1 to 3, 48 beyond.
template <class F>
void with_width(int dim, F f) {
    if (dim <= 10) f(std::integral_constant<int, 10>{});
    else if (dim <= 24) f(std::integral_constant<int, 24>{});
    else if (dim <= 46) f(std::integral_constant<int, 46>{});
    else f(std::integral_constant<int, kCbMaxDim>{});
}

// (In this namespace, so that the library has its own `attr`: a static of a template with a name for the linker is one
// object of the process, also when a release and a debug library are loaded, each with kernels of its own.)
template <int DIM>
cudaError_t launch_assign_tc(const float *pts, int64_t n, int dim, int64_t stride, const float *cent, int k,
                             uint32_t *assign, cudaStream_t st) {
    constexpr size_t smem = sizeof(TcSmem) + 1024;
    static PerDevice attr;
    attr.get([] {
        cudaFuncSetAttribute(k_kmeans_assign_tc<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
        return 1;
    });
    k_kmeans_assign_tc<DIM><<<static_cast<unsigned>((n + kTcPoints - 1) / kTcPoints), kTcThreads, smem, st>>>(
        pts, n, dim, stride, cent, k, assign);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_kmeans_assign(const float *pts, int64_t n, int dim, int64_t stride, const float *cent, int k,
                                 uint32_t *assign, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (k >= kTcMinCentroids && n >= kTcMinPoints) {
        const cudaError_t e = dim == 45   ? launch_assign_tc<45>(pts, n, dim, stride, cent, k, assign, st)
                              : dim == 24 ? launch_assign_tc<24>(pts, n, dim, stride, cent, k, assign, st)
                              : dim == 9  ? launch_assign_tc<9>(pts, n, dim, stride, cent, k, assign, st)
                                          : launch_assign_tc<0>(pts, n, dim, stride, cent, k, assign, st);
        if (e != cudaSuccess) return e;
        with_width(dim, [&](auto d) {
            k_kmeans_assign_left<decltype(d)::value>
                <<<static_cast<unsigned>((n + kLeftPoints - 1) / kLeftPoints), kLeftPoints, 0, st>>>(pts, n, dim, stride, cent,
                                                                                                     k, assign);
        });
        return cudaGetLastError();
    }
    with_width(dim, [&](auto d) {
        k_kmeans_assign<decltype(d)::value><<<static_cast<unsigned>((n + kKmThreads - 1) / kKmThreads), kKmThreads, 0, st>>>(
            pts, n, dim, stride, cent, k, assign);
    });
    return cudaGetLastError();
}

cudaError_t launch_kmeans_update(const float *pts, int64_t n, int dim, int64_t stride, const uint32_t *assign, int k,
                                 float *cent, float *scratch, cudaStream_t st) {
    float *sums = scratch, *cnt = scratch + static_cast<size_t>(k) * dim;
    cudaError_t e = cudaMemsetAsync(scratch, 0, static_cast<size_t>(k) * (dim + 1) * sizeof(float), st);
    if (e != cudaSuccess) return e;
    if (n > 0) {
        const int blocks = static_cast<int>(std::min<int64_t>((n + 31) / 32, 8 * 1024));
        k_kmeans_accumulate<<<blocks, 256, 0, st>>>(pts, n, dim, stride, assign, sums, cnt);
    }
    const int64_t tot = static_cast<int64_t>(k) * dim;
    k_kmeans_finish<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(sums, cnt, k, dim, cent);
    return cudaGetLastError();
}

cudaError_t launch_sh_encode(const float *sh, int64_t n, int K, const uint32_t *assign, const float *cent, int k,
                             float *dc, uint16_t *index, void *table, cudaStream_t st) {
    const int row = cb_row_halves(K);
    const int64_t tot = std::max<int64_t>(n, static_cast<int64_t>(k) * row);
    if (tot == 0) return cudaSuccess;
    k_sh_encode<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(sh, n, K, assign, cent, k, row, dc, index,
                                                                       static_cast<__half *>(table));
    return cudaGetLastError();
}

}  // namespace gs

extern "C" int gs_debug_kmeans_wait(uint32_t limit) {
#ifdef GS_DEBUG
    const uint32_t v = limit ? limit : gs::kTcWaitLimit;
    const cudaError_t e = cudaMemcpyToSymbol(gs::g_dbg_tc_wait, &v, sizeof v);
    return e == cudaSuccess ? GS_OK : gs::report(GS_ERR_CUDA, cudaGetErrorString(e));
#else
    (void)limit;
    return gs::report(GS_ERR_INVALID, "gs_debug_kmeans_wait: only in GS_DEBUG builds");
#endif
}
