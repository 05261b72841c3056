// S1 - per-Gaussian preprocess: layer-mask / clip-plane / near culls, EWA
// projection (Sec. 2.2.1), exponent coefficients, SH colour, opacity, tile
// rectangle and depth key (Sec. 3.3: only active layers are drawn; Gaussians
// sorted relative to the camera).
//
// This translation unit is compiled with -fmad=false: every a*b+c below is a
// rounded multiply followed by a rounded add, evaluated in the written order,
// so the integer decisions (culls, radius, rectangle, depth bits) are a fixed
// function of the float32 inputs (bit-exact tile ids and sort order).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "gs_internal.cuh"

namespace gs {
namespace {

// exp(x) by Cody-Waite range reduction (x = k ln2 + r, ln2 split in a 16-bit
// head and a tail; Cody & Waite 1980) and the degree-7 Taylor series of exp(r)
// in Horner form.  Only +, -, * and an exact power-of-two scaling are used, so
// the result is reproducible on any IEEE single-precision machine.
__device__ __forceinline__ float exp_cw(float x) {
    x = fminf(fmaxf(x, -80.0f), 80.0f);
    float k = rintf(x * 0x1.715476p+0f);
    float r = (x - k * 0x1.62e4p-1f) - k * 0x1.7f7d1cp-20f;
    float p = 0x1.a01a02p-13f;
    p = p * r + 0x1.6c16c2p-10f;
    p = p * r + 0x1.111112p-7f;
    p = p * r + 0x1.555556p-5f;
    p = p * r + 0x1.555556p-3f;
    p = p * r + 0.5f;
    p = p * r + 1.0f;
    p = p * r + 1.0f;
    return p * __int_as_float((static_cast<int>(k) + 127) << 23);
}

__device__ __forceinline__ float ld_half(const void *p, int64_t idx, int dtype) {
    if (dtype == GS_DTYPE_F16) return __half2float(static_cast<const __half *>(p)[idx]);
    if (dtype == GS_DTYPE_BF16) return __bfloat162float(static_cast<const __nv_bfloat16 *>(p)[idx]);
    return static_cast<const float *>(p)[idx];
}

// Four consecutive 16-bit values.
__device__ __forceinline__ void widen4(uint2 v, int dtype, float *o) {
    if (dtype == GS_DTYPE_F16) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
        o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
    } else {                                                // bf16: the upper half of a float
        o[0] = __uint_as_float(v.x << 16); o[1] = __uint_as_float(v.x & 0xFFFF0000u);
        o[2] = __uint_as_float(v.y << 16); o[3] = __uint_as_float(v.y & 0xFFFF0000u);
    }
}

// Real SH basis (Condon-Shortley phase, index l*l+l+m) from the textbook
// Cartesian forms; constants are the float nearest the exact normalisations.
template <int deg>
__device__ __forceinline__ void sh_basis(float x, float y, float z, float *b) {
    b[0] = 0x1.20dd76p-2f;                                  // 1/(2 sqrt(pi))
    if constexpr (deg < 1) return;
    const float C1 = 0x1.f45438p-2f;                        // sqrt(3/(4 pi))
    b[1] = -C1 * y;
    b[2] = C1 * z;
    b[3] = -C1 * x;
    if constexpr (deg < 2) return;
    const float C2A = 0x1.17b142p+0f, C2C = 0x1.42f602p-2f, C2E = 0x1.17b142p-1f;
    float xx = x * x, yy = y * y, zz = z * z, xy = x * y, yz = y * z, xz = x * z;
    b[4] = C2A * xy;
    b[5] = -C2A * yz;
    b[6] = C2C * ((2.0f * zz - xx) - yy);
    b[7] = -C2A * xz;
    b[8] = C2E * (xx - yy);
    if constexpr (deg < 3) return;
    const float C3A = 0x1.2e1a32p-1f, C3B = 0x1.71ff8ep+1f, C3C = 0x1.d403d0p-2f, C3D = 0x1.7e21f0p-2f,
                C3F = 0x1.71ff8ep+0f;
    b[9] = (-C3A * y) * (3.0f * xx - yy);
    b[10] = (C3B * xy) * z;
    b[11] = (-C3C * y) * ((4.0f * zz - xx) - yy);
    b[12] = (C3D * z) * ((2.0f * zz - 3.0f * xx) - 3.0f * yy);
    b[13] = (-C3C * x) * ((4.0f * zz - xx) - yy);
    b[14] = (C3F * z) * (xx - yy);
    b[15] = (-C3A * x) * (xx - 3.0f * yy);
}

__device__ __forceinline__ void store_geo(Geo *g, const float4 a, const float4 b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// Several views of one launch: with ONE they show the same scene and a thread
// takes its Gaussian through all of them, so what does not depend on the view
// (exponentials, rotation, covariance, opacity) is computed once; otherwise
// the views are interleaved block by block (view blockIdx.x mod n).
template <int DEG, int NV, bool ONE>
__global__ void __launch_bounds__(128) k_preprocess(const __grid_constant__ Views<PreView, NV> B) {
    chain_start();
    const int view = ONE ? 0 : blockIdx.x % B.n;
    const SceneView &s = B[view].s;
    const int i = (NV == 1 || ONE ? blockIdx.x : blockIdx.x / B.n) * blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int lay = s.layer[i];
    const float mx = s.means[3 * i], my = s.means[3 * i + 1], mz = s.means[3 * i + 2];
    // the other per-Gaussian inputs but SH, loaded with these before the culling tests so that one memory
    // latency covers them all
    const float ls0 = ld_half(s.log_scales, 3 * (int64_t)i, s.dtype_sr);
    const float ls1 = ld_half(s.log_scales, 3 * (int64_t)i + 1, s.dtype_sr);
    const float ls2 = ld_half(s.log_scales, 3 * (int64_t)i + 2, s.dtype_sr);
    float qw, qx, qy, qz;
    if (s.dtype_sr == GS_DTYPE_F32) {
        const float4 q = reinterpret_cast<const float4 *>(s.quats)[i];
        qw = q.x; qx = q.y; qy = q.z; qz = q.w;
    } else {
        float q[4];
        widen4(reinterpret_cast<const uint2 *>(s.quats)[i], s.dtype_sr, q);
        qw = q[0]; qx = q[1]; qy = q[2]; qz = q[3];
    }
    const float ol = s.opacity_logit[i];
    // not masked, not clipped and in front of the view's near plane
    const auto kept = [&](const PreView &V) {
        const Planes &pl = V.pl;
        const float *R = V.c.R;
        bool keep = (V.layer_mask >> lay) & 1u;
        for (int k = 0; k < pl.n && keep; ++k) {
            if (!((pl.bits[k] >> lay) & 1u)) continue;
            const float4 p = pl.p[k];
            const float dist = ((p.x * mx + p.y * my) + p.z * mz) + p.w;
            if (dist < 0.0f) keep = false;
        }
        const float pz = ((R[6] * mx + R[7] * my) + R[8] * mz) + V.c.t[2];
        return keep && pz > V.c.znear;
    };
    bool some;                                     // kept in the view, or for several: on in one of them
    if constexpr (ONE) {
        uint32_t layers = 0;
        for (int v = 0; v < B.n; ++v) layers |= B[v].layer_mask;
        some = (layers >> lay) & 1u;
    } else {
        some = kept(B[view]);
    }
    float S00 = 0.f, S01 = 0.f, S02 = 0.f, S11 = 0.f, S12 = 0.f, S22 = 0.f, opac = 0.f;
    if (some) {
        // the SH row (read only if the splat turns out visible) is brought into L2 while the projection runs
        if (s.dtype_sh != GS_DTYPE_SH_CODEBOOK) {
            constexpr int K = (DEG + 1) * (DEG + 1);
            const int bytes = 3 * K * (s.dtype_sh == GS_DTYPE_F32 ? 4 : 2);
            const char *row = static_cast<const char *>(s.sh) + static_cast<int64_t>(i) * bytes;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(row));                  // first and last byte of the
            asm volatile("prefetch.global.L2 [%0];" ::"l"(row + bytes - 1));      // row: its one or two lines
        }
        const float s0 = exp_cw(ls0);
        const float s1 = exp_cw(ls1);
        const float s2 = exp_cw(ls2);
        const float qq = ((qw * qw + qx * qx) + qy * qy) + qz * qz;
        const float qn = sqrtf(qq);
        const float w = qw / qn, x = qx / qn, y = qy / qn, z = qz / qn;
        const float r00 = 1.0f - 2.0f * (y * y + z * z), r01 = 2.0f * (x * y - w * z), r02 = 2.0f * (x * z + w * y);
        const float r10 = 2.0f * (x * y + w * z), r11 = 1.0f - 2.0f * (x * x + z * z), r12 = 2.0f * (y * z - w * x);
        const float r20 = 2.0f * (x * z - w * y), r21 = 2.0f * (y * z + w * x), r22 = 1.0f - 2.0f * (x * x + y * y);
        const float m00 = r00 * s0, m01 = r01 * s1, m02 = r02 * s2;
        const float m10 = r10 * s0, m11 = r11 * s1, m12 = r12 * s2;
        const float m20 = r20 * s0, m21 = r21 * s1, m22 = r22 * s2;
        S00 = (m00 * m00 + m01 * m01) + m02 * m02;
        S01 = (m00 * m10 + m01 * m11) + m02 * m12;
        S02 = (m00 * m20 + m01 * m21) + m02 * m22;
        S11 = (m10 * m10 + m11 * m11) + m12 * m12;
        S12 = (m10 * m20 + m11 * m21) + m12 * m22;
        S22 = (m20 * m20 + m21 * m21) + m22 * m22;
        opac = 1.0f / (1.0f + exp_cw(-ol));
    }
    const auto project = [&](const PreView &V) {
        const CamView &c = V.c;
        uint32_t ntiles = 0;
        uint32_t dkey = 0xFFFFFFFFu;
        const float *R = c.R;
        const float pz = ((R[6] * mx + R[7] * my) + R[8] * mz) + c.t[2];
        if (ONE ? kept(V) : some) {
            const float px = ((R[0] * mx + R[1] * my) + R[2] * mz) + c.t[0];
            const float py = ((R[3] * mx + R[4] * my) + R[5] * mz) + c.t[1];
            const float limx = kFrustumClamp * ((0.5f * static_cast<float>(c.W)) / c.fx);
            const float limy = kFrustumClamp * ((0.5f * static_cast<float>(c.H)) / c.fy);
            const float izx = px / pz, izy = py / pz;
            const float cxz = fminf(limx, fmaxf(-limx, izx));
            const float cyz = fminf(limy, fmaxf(-limy, izy));
            const float j00 = c.fx / pz, j02 = -(c.fx * cxz) / pz;
            const float j11 = c.fy / pz, j12 = -(c.fy * cyz) / pz;
            const float t00 = j00 * R[0] + j02 * R[6], t01 = j00 * R[1] + j02 * R[7], t02 = j00 * R[2] + j02 * R[8];
            const float t10 = j11 * R[3] + j12 * R[6], t11 = j11 * R[4] + j12 * R[7], t12 = j11 * R[5] + j12 * R[8];
            const float u00 = (t00 * S00 + t01 * S01) + t02 * S02;
            const float u01 = (t00 * S01 + t01 * S11) + t02 * S12;
            const float u02 = (t00 * S02 + t01 * S12) + t02 * S22;
            const float u10 = (t10 * S00 + t11 * S01) + t12 * S02;
            const float u11 = (t10 * S01 + t11 * S11) + t12 * S12;
            const float u12 = (t10 * S02 + t11 * S12) + t12 * S22;
            const float c00 = ((u00 * t00 + u01 * t01) + u02 * t02) + kDilation;
            const float c01 = (u00 * t10 + u01 * t11) + u02 * t12;
            const float c11 = ((u10 * t10 + u11 * t11) + u12 * t12) + kDilation;
            const float det = c00 * c11 - c01 * c01;
            if (det > 0.0f) {
                const float mid = 0.5f * (c00 + c11);
                const float disc = fmaxf(kEigenFloor, mid * mid - det);
                const float lam = mid + sqrtf(disc);
                const float r = ceilf(kRadiusSigmas * sqrtf(lam));
                const float uu = c.fx * izx + c.cx, vv = c.fy * izy + c.cy;
                const float fTx = static_cast<float>(c.Tx), fTy = static_cast<float>(c.Ty);
                const float fx0 = fminf(fTx, fmaxf(0.0f, truncf((uu - r) * 0.0625f)));
                const float fy0 = fminf(fTy, fmaxf(0.0f, truncf((vv - r) * 0.0625f)));
                const float fx1 = fminf(fTx, fmaxf(0.0f, truncf(((uu + r) + 15.0f) * 0.0625f)));
                const float fy1 = fminf(fTy, fmaxf(0.0f, truncf(((vv + r) + 15.0f) * 0.0625f)));
                const int x0 = static_cast<int>(fx0), y0 = static_cast<int>(fy0);
                const int x1 = static_cast<int>(fx1), y1 = static_cast<int>(fy1);
                ntiles = GS_CHECK(x0 <= x1 && y0 <= y1 && x1 <= c.Tx && y1 <= c.Ty, V.ctl, kSiteRect)
                             ? static_cast<uint32_t>((x1 - x0) * (y1 - y0))
                             : 0u;
                if (ntiles > 0) {
                    // view-dependent colour
                    const float campos0 = -((R[0] * c.t[0] + R[3] * c.t[1]) + R[6] * c.t[2]);
                    const float campos1 = -((R[1] * c.t[0] + R[4] * c.t[1]) + R[7] * c.t[2]);
                    const float campos2 = -((R[2] * c.t[0] + R[5] * c.t[1]) + R[8] * c.t[2]);
                    const float dx = mx - campos0, dy = my - campos1, dz = mz - campos2;
                    const float dn = sqrtf((dx * dx + dy * dy) + dz * dz);
                    constexpr int K = (DEG + 1) * (DEG + 1);
                    float b[K];
                    sh_basis<DEG>(dx / dn, dy / dn, dz / dn, b);
                    const int64_t base = static_cast<int64_t>(i) * K * 3;
                    float shv[3 * K];
                    if (s.dtype_sh == GS_DTYPE_SH_CODEBOOK) {
                        // DC per Gaussian; coefficients k >= 1 from the FP16 table row (16-byte loads from L2)
                        const float *dcp = static_cast<const float *>(s.sh) + static_cast<int64_t>(i) * 3;
                        shv[0] = dcp[0]; shv[1] = dcp[1]; shv[2] = dcp[2];
                        constexpr int ROW = cb_row_halves(K);
                        const uint4 *row = reinterpret_cast<const uint4 *>(static_cast<const __half *>(s.sh_table) +
                                                                           static_cast<int64_t>(s.sh_index[i]) * ROW);
#pragma unroll
                        for (int q = 0; q < ROW / 8; ++q) {
                            const uint4 v = row[q];
                            const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                const float2 f = __half22float2(h[r]);
                                const int d0 = 8 * q + 2 * r;
                                if (d0 < 3 * (K - 1)) shv[3 + d0] = f.x;
                                if (d0 + 1 < 3 * (K - 1)) shv[3 + d0 + 1] = f.y;
                            }
                        }
                    } else if (s.dtype_sh == GS_DTYPE_F32 && (3 * K) % 4 == 0) {
                        // 16-byte loads of this Gaussian's coefficients (its row starts 16-byte aligned)
                        const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(s.sh) + base);
#pragma unroll
                        for (int k = 0; k < 3 * K / 4; ++k) {
                            const float4 v = src[k];
                            shv[4 * k] = v.x; shv[4 * k + 1] = v.y; shv[4 * k + 2] = v.z; shv[4 * k + 3] = v.w;
                        }
                    } else if (s.dtype_sh != GS_DTYPE_F32 && (3 * K) % 4 == 0) {
                        // 16-bit storage: rows of 96 bytes in 16-byte loads, of 24 in 8-byte ones (one coefficient at a
                        // time: 1.5M Gaussians 0.076 ms against 0.062)
                        const uint16_t *src = static_cast<const uint16_t *>(s.sh) + base;
                        if constexpr ((3 * K) % 8 == 0) {
#pragma unroll
                            for (int k = 0; k < 3 * K / 8; ++k) {
                                const uint4 v = reinterpret_cast<const uint4 *>(src)[k];
                                widen4(make_uint2(v.x, v.y), s.dtype_sh, shv + 8 * k);
                                widen4(make_uint2(v.z, v.w), s.dtype_sh, shv + 8 * k + 4);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 3 * K / 4; ++k)
                                widen4(reinterpret_cast<const uint2 *>(src)[k], s.dtype_sh, shv + 4 * k);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 3 * K; ++k) shv[k] = ld_half(s.sh, base + k, s.dtype_sh);
                    }
                    float rgb[3];
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        float acc = b[0] * shv[ch];
#pragma unroll
                        for (int k = 1; k < K; ++k) acc = acc + b[k] * shv[3 * k + ch];
                        rgb[ch] = fmaxf(acc + 0.5f, 0.0f);
                    }
                    const float NHL = -0x1.715476p-1f;   // -log2(e)/2
                    Rec o;
                    o.a = make_float4(uu, vv, (c11 / det) * NHL, -(c01 / c11));
                    o.b = make_float4(NHL / c11, opac, rgb[0], rgb[1]);
                    o.c = make_float4(rgb[2], pz, __uint_as_float(static_cast<uint32_t>(x0) | (static_cast<uint32_t>(y0) << 16)),
                                      __uint_as_float(static_cast<uint32_t>(x1) | (static_cast<uint32_t>(y1) << 16)));
                    V.rec[i] = o;
                    store_geo(V.geo + i, o.a, o.b);
                    dkey = __float_as_uint(pz);
                }
            }
        }
        V.tiles[i] = ntiles;
        V.depth[i] = dkey;
    };
    if constexpr (ONE) {
#pragma unroll 1
        for (int v = 0; v < B.n; ++v) project(B[v]);
    } else {
        project(B[view]);
    }
}

// Zeroes every view's control block and what is cleared with it (16-byte words).
template <int NV>
__global__ void __launch_bounds__(256) k_clear(const __grid_constant__ Views<PreView, NV> B) {
    chain_start();
    const PreView &V = B[blockIdx.y];
    uint4 *p = reinterpret_cast<uint4 *>(V.ctl);
    const size_t words = V.clear_bytes / sizeof(uint4);
    for (size_t w = blockIdx.x * 256u + threadIdx.x; w < words; w += gridDim.x * 256u) p[w] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

namespace {

template <int NV, bool ONE>
void preprocess_views(int deg, const Views<PreView, NV> &b, unsigned blocks, cudaStream_t st) {
    switch (deg) {
        case 0: launch_chained(k_preprocess<0, NV, ONE>, blocks, 128, 0, st, b); break;
        case 1: launch_chained(k_preprocess<1, NV, ONE>, blocks, 128, 0, st, b); break;
        case 2: launch_chained(k_preprocess<2, NV, ONE>, blocks, 128, 0, st, b); break;
        default: launch_chained(k_preprocess<3, NV, ONE>, blocks, 128, 0, st, b); break;
    }
}

}  // namespace

cudaError_t launch_clear(const PreView *views, int n, cudaStream_t st) {
    size_t most = 0;
    for (int i = 0; i < n; ++i) most = views[i].clear_bytes > most ? views[i].clear_bytes : most;
    // four 16-byte words a thread, at most a block per SM
    const size_t want = (most + 256 * 64 - 1) / (256 * 64);
    const unsigned blocks = static_cast<unsigned>(want < 152 ? want : 152);
    with_views(views, n, [&](const auto &b) {
        constexpr int NV = sizeof(b.v) / sizeof(PreView);
        k_clear<NV><<<dim3(blocks, b.n), 256, 0, st>>>(b);       // (whatever ran before is waited for as usual)
    });
    return cudaGetLastError();
}

// Gaussians times views from which views of one scene are taken together; below, the blocks of one view leave SMs
// idle.  Degree 3, two views of 131,072 Gaussians 22.6 against 20.6 us view by view, of 262,144 34.0 against 34.8;
// eight views of 32,000 23.0 against 20.5, of 65,000 31.6 against 33.4, of 262,144 88.5 against 110.7, of 500,000
// 155 against 199; the two eyes of the 3M-Gaussian stereo pair 120 against 131.
constexpr int64_t kSharedMin = 1 << 19;

bool same_scene(const SceneView &a, const SceneView &b) {
    return a.means == b.means && a.log_scales == b.log_scales && a.quats == b.quats &&
           a.opacity_logit == b.opacity_logit && a.sh == b.sh && a.layer == b.layer && a.sh_index == b.sh_index &&
           a.sh_table == b.sh_table && a.sh_table_rows == b.sh_table_rows && a.n == b.n &&
           a.sh_degree == b.sh_degree && a.dtype_sh == b.dtype_sh && a.dtype_sr == b.dtype_sr;
}

cudaError_t launch_preprocess(const PreView *views, int n, cudaStream_t st, int *launches) {
    *launches = 0;
    for (int deg = 0; deg <= 3; ++deg) {           // a launch per SH degree among the views
        PreView of[kMaxBatch];
        int m = 0, most = 0;
        for (int i = 0; i < n && m < kMaxBatch; ++i) {
            if (views[i].s.sh_degree != deg || views[i].s.n == 0) continue;
            of[m++] = views[i];
            most = views[i].s.n > most ? views[i].s.n : most;
        }
        if (m == 0) continue;
        bool one = m > 1 && static_cast<int64_t>(most) * m >= kSharedMin;
        for (int i = 1; i < m; ++i) one = one && same_scene(of[0].s, of[i].s);
        const unsigned blocks = static_cast<unsigned>((most + 127) / 128);
        with_views(of, m, [&](const auto &b) {
            constexpr int NV = sizeof(b.v) / sizeof(PreView);
            if (one) preprocess_views<NV, NV != 1>(deg, b, blocks, st);
            else preprocess_views<NV, false>(deg, b, blocks * static_cast<unsigned>(m), st);
        });
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace gs
