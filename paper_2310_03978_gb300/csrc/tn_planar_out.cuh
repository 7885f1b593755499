// Device store of the direct planar output (PlanarOut, declared in tn_internal.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tn_internal.h"

namespace tn {

// FP32 rounded to the nearest TF32 value (10 fraction bits, ties away from zero), kept in an
// FP32 container: the tensor core then reads it without further rounding.
__device__ __forceinline__ float round_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// N = 2, 4 or 8 consecutive complex values (offset off a multiple of N) into a TF32 planar output:
// one 8-byte word, or 16-byte words, per plane.  A power-of-two scale does not change TF32's (or
// BF16's) significand, so the values a tensor core reads are those a conversion pass would write,
// up to that scale.
template <int N, bool SCALE>
__device__ __forceinline__ void planar_out_store_tf32(const PlanarOut &o, int64_t s, uint64_t off,
                                                      const float2 (&v)[N], int e) {
    const Pow2 pe = pow2_of(-e);
    float *base = static_cast<float *>(o.base) + s * o.sstride + (int64_t)off;
    float p[4][N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float r = SCALE ? scale_pow2(v[j].x, pe) : v[j].x;
        const float i = SCALE ? scale_pow2(v[j].y, pe) : v[j].y;
        p[0][j] = round_tf32(r);
        p[1][j] = round_tf32(i);
        if (o.planes == 3) p[2][j] = round_tf32(r + i);
        if (o.planes == 4) {
            p[2][j] = round_tf32(r - p[0][j]);
            p[3][j] = round_tf32(i - p[1][j]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (q >= o.planes) break;
        float *d = base + q * o.plane_stride;
        if constexpr (N == 2) {
            *reinterpret_cast<float2 *>(d) = make_float2(p[q][0], p[q][1]);
        } else {
#pragma unroll
            for (int j = 0; j < N; j += 4)
                *reinterpret_cast<float4 *>(d + j) =
                    make_float4(p[q][j], p[q][j + 1], p[q][j + 2], p[q][j + 3]);
        }
    }
}

// Store two adjacent complex values (offsets off and off + 1, off even) into the planar output
// as one 2 x 16-bit word per plane.
__device__ __forceinline__ void planar_out_store2(const PlanarOut &o, int64_t s, uint64_t off,
                                                  float2 v0, float2 v1, int e) {
    if (o.dtype == 2) {
        const float2 v[2] = {v0, v1};
        planar_out_store_tf32<2, true>(o, s, off, v, e);
        return;
    }
    const Pow2 pe = pow2_of(-e);
    const float r0 = scale_pow2(v0.x, pe), i0 = scale_pow2(v0.y, pe);
    const float r1 = scale_pow2(v1.x, pe), i1 = scale_pow2(v1.y, pe);
    const int64_t base = s * o.sstride + (int64_t)off;
    const int64_t ps = o.plane_stride / 2;
    if (o.dtype == 1) {
        __nv_bfloat162 *p =
            reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(o.base) + base);
        const __nv_bfloat162 rh = __floats2bfloat162_rn(r0, r1), ih = __floats2bfloat162_rn(i0, i1);
        p[0] = rh;
        p[ps] = ih;
        if (o.planes == 3) p[2 * ps] = __floats2bfloat162_rn(r0 + i0, r1 + i1);
        if (o.planes == 4) {
            const float2 rf = __bfloat1622float2(rh), jf = __bfloat1622float2(ih);
            p[2 * ps] = __floats2bfloat162_rn(r0 - rf.x, r1 - rf.y);
            p[3 * ps] = __floats2bfloat162_rn(i0 - jf.x, i1 - jf.y);
        }
    } else {
        __half2 *p = reinterpret_cast<__half2 *>(static_cast<__half *>(o.base) + base);
        const __half2 rh = __floats2half2_rn(r0, r1), ih = __floats2half2_rn(i0, i1);
        p[0] = rh;
        p[ps] = ih;
        if (o.planes == 3) p[2 * ps] = __floats2half2_rn(r0 + i0, r1 + i1);
        if (o.planes == 4) {
            const float2 rf = __half22float2(rh), jf = __half22float2(ih);
            p[2 * ps] = __floats2half2_rn(r0 - rf.x, r1 - rf.y);
            p[3 * ps] = __floats2half2_rn(i0 - jf.x, i1 - jf.y);
        }
    }
}

// Store eight consecutive complex values (offsets off .. off + 7, off a multiple of 8) into the
// planar output as one 16-byte word (8 x 16 bits) per plane.
template <typename T2>
__device__ __forceinline__ T2 pack_pair(float a, float b);
template <>
__device__ __forceinline__ __half2 pack_pair<__half2>(float a, float b) {
    return __floats2half2_rn(a, b);
}
template <>
__device__ __forceinline__ __nv_bfloat162 pack_pair<__nv_bfloat162>(float a, float b) {
    return __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ float2 unpack_pair(__half2 h) { return __half22float2(h); }
__device__ __forceinline__ float2 unpack_pair(__nv_bfloat162 h) { return __bfloat1622float2(h); }

template <typename T2, bool SCALE>
__device__ __forceinline__ void planar_out_store8_t(const PlanarOut &o, int64_t s, uint64_t off,
                                                    const float2 (&v)[8], int e) {
    union Row {
        uint4 u;
        T2 h[4];
    } re, im, p2, p3;
    const Pow2 pe = pow2_of(-e);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float r0 = SCALE ? scale_pow2(v[2 * j].x, pe) : v[2 * j].x;
        const float i0 = SCALE ? scale_pow2(v[2 * j].y, pe) : v[2 * j].y;
        const float r1 = SCALE ? scale_pow2(v[2 * j + 1].x, pe) : v[2 * j + 1].x;
        const float i1 = SCALE ? scale_pow2(v[2 * j + 1].y, pe) : v[2 * j + 1].y;
        re.h[j] = pack_pair<T2>(r0, r1);
        im.h[j] = pack_pair<T2>(i0, i1);
        if (o.planes == 3) p2.h[j] = pack_pair<T2>(r0 + i0, r1 + i1);
        if (o.planes == 4) {
            const float2 rf = unpack_pair(re.h[j]), jf = unpack_pair(im.h[j]);
            p2.h[j] = pack_pair<T2>(r0 - rf.x, r1 - rf.y);
            p3.h[j] = pack_pair<T2>(i0 - jf.x, i1 - jf.y);
        }
    }
    uint16_t *base = static_cast<uint16_t *>(o.base) + s * o.sstride + (int64_t)off;
    *reinterpret_cast<uint4 *>(base) = re.u;
    *reinterpret_cast<uint4 *>(base + o.plane_stride) = im.u;
    if (o.planes >= 3) *reinterpret_cast<uint4 *>(base + 2 * o.plane_stride) = p2.u;
    if (o.planes == 4) *reinterpret_cast<uint4 *>(base + 3 * o.plane_stride) = p3.u;
}

// Store four consecutive complex values (offsets off .. off + 3, off a multiple of 4) into the
// planar output as one 8-byte word (4 x 16 bits) per plane.
template <typename T2>
__device__ __forceinline__ void planar_out_store4_t(const PlanarOut &o, int64_t s, uint64_t off,
                                                    const float2 (&v)[4], int e) {
    union Half {
        uint2 u;
        T2 h[2];
    } re, im, p2, p3;
    const Pow2 pe = pow2_of(-e);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float r0 = scale_pow2(v[2 * j].x, pe), i0 = scale_pow2(v[2 * j].y, pe);
        const float r1 = scale_pow2(v[2 * j + 1].x, pe), i1 = scale_pow2(v[2 * j + 1].y, pe);
        re.h[j] = pack_pair<T2>(r0, r1);
        im.h[j] = pack_pair<T2>(i0, i1);
        if (o.planes == 3) p2.h[j] = pack_pair<T2>(r0 + i0, r1 + i1);
        if (o.planes == 4) {
            const float2 rf = unpack_pair(re.h[j]), jf = unpack_pair(im.h[j]);
            p2.h[j] = pack_pair<T2>(r0 - rf.x, r1 - rf.y);
            p3.h[j] = pack_pair<T2>(i0 - jf.x, i1 - jf.y);
        }
    }
    uint16_t *base = static_cast<uint16_t *>(o.base) + s * o.sstride + (int64_t)off;
    *reinterpret_cast<uint2 *>(base) = re.u;
    *reinterpret_cast<uint2 *>(base + o.plane_stride) = im.u;
    if (o.planes >= 3) *reinterpret_cast<uint2 *>(base + 2 * o.plane_stride) = p2.u;
    if (o.planes == 4) *reinterpret_cast<uint2 *>(base + 3 * o.plane_stride) = p3.u;
}

// ESZ: bytes of a stored number, 2 (FP16 or BF16 by o.dtype) or 4 (TF32).
template <int ESZ>
__device__ __forceinline__ void planar_out_store4(const PlanarOut &o, int64_t s, uint64_t off,
                                                  const float2 (&v)[4], int e) {
    if constexpr (ESZ == 4) planar_out_store_tf32<4, true>(o, s, off, v, e);
    else if (o.dtype == 1) planar_out_store4_t<__nv_bfloat162>(o, s, off, v, e);
    else planar_out_store4_t<__half2>(o, s, off, v, e);
}

template <int ESZ>
__device__ __forceinline__ void planar_out_store8(const PlanarOut &o, int64_t s, uint64_t off,
                                                  const float2 (&v)[8], int e) {
    if constexpr (ESZ == 4) planar_out_store_tf32<8, true>(o, s, off, v, e);
    else if (o.dtype == 1) planar_out_store8_t<__nv_bfloat162, true>(o, s, off, v, e);
    else planar_out_store8_t<__half2, true>(o, s, off, v, e);
}

// The same for values already multiplied by 2^-e.
template <int ESZ>
__device__ __forceinline__ void planar_out_store8_prescaled(const PlanarOut &o, int64_t s,
                                                            uint64_t off, const float2 (&v)[8]) {
    if constexpr (ESZ == 4) planar_out_store_tf32<8, false>(o, s, off, v, 0);
    else if (o.dtype == 1) planar_out_store8_t<__nv_bfloat162, false>(o, s, off, v, 0);
    else planar_out_store8_t<__half2, false>(o, s, off, v, 0);
}

}  // namespace tn
