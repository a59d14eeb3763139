// Packed fp32 channel arithmetic of the edge kernels.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace dmts {

// ------------------------------------------------------------ channel packs
// A lane owns CPW consecutive channels. With CPW even they are processed as
// pairs in packed fp32 arithmetic (fma.rn.f32x2 / mul.rn.f32x2 of sm_100 and
// later: one instruction issues two channels, each element rounded exactly as
// fmaf / a plain product), with CPW = 1 as scalars. Quantities that multiply
// every channel alike (radial basis, harmonics) are stored in shared memory
// already duplicated into both halves of a pair.
template <int CPW>
struct Pack {
    static constexpr int W = CPW % 2 == 0 ? 2 : 1;   // channels per pack
    static constexpr int NP = CPW / W;               // packs per lane
    using T = typename std::conditional<W == 2, float2, float>::type;
};

__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vsum(float2 v) { return v.x + v.y; }
__device__ __forceinline__ float vsum(float v) { return v; }
__device__ __forceinline__ float vget(float2 v, int h) { return h ? v.y : v.x; }
__device__ __forceinline__ float vget(float v, int) { return v; }
template <class T>
__device__ __forceinline__ T vdup(float v) {
    if constexpr (std::is_same<T, float2>::value) return make_float2(v, v);
    else return v;
}

template <class T>
__device__ __forceinline__ T vpair(float a, float b) {
    if constexpr (std::is_same<T, float2>::value) return make_float2(a, b);
    else return a;
}

// CPW consecutive floats at p (aligned to 4 * CPW bytes) as packs, and back.
template <int CPW, class T>
__device__ __forceinline__ void ldp(const float *p, T *v) {
    if constexpr (CPW == 4) {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = make_float2(t.x, t.y);
        v[1] = make_float2(t.z, t.w);
    } else if constexpr (CPW == 2) {
        v[0] = __ldg(reinterpret_cast<const float2 *>(p));
    } else {
        v[0] = __ldg(p);
    }
}

// The same from shared memory.
template <int CPW, class T>
__device__ __forceinline__ void ldp_s(const float *p, T *v) {
    if constexpr (CPW == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = make_float2(t.x, t.y);
        v[1] = make_float2(t.z, t.w);
    } else if constexpr (CPW == 2) {
        v[0] = *reinterpret_cast<const float2 *>(p);
    } else {
        v[0] = *p;
    }
}

template <int CPW, class T>
__device__ __forceinline__ void stp(float *p, const T *v) {
    if constexpr (CPW == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    else if constexpr (CPW == 2) *reinterpret_cast<float2 *>(p) = v[0];
    else *p = v[0];
}

// CPW consecutive channels from column c of row r of a split-bf16 copy with
// logical row length N (common.cuh): one store for the hi parts, one for the
// lo parts.
template <int CPW, int PW, class T>
__device__ __forceinline__ void st_split_p(__nv_bfloat16 *base, size_t r, int N, int c, const T *v) {
    uint16_t h[CPW], l[CPW];
#pragma unroll
    for (int u = 0; u < CPW; ++u) {
        __nv_bfloat16 hi, lo;
        split_bf16(vget(v[u / PW], u % PW), hi, lo);
        h[u] = __bfloat16_as_ushort(hi);
        l[u] = __bfloat16_as_ushort(lo);
    }
    __nv_bfloat16 *p = base + r * 2 * N + c;
    if constexpr (CPW == 4) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16);
        *reinterpret_cast<uint2 *>(p + N) = make_uint2(l[0] | (uint32_t)l[1] << 16, l[2] | (uint32_t)l[3] << 16);
    } else if constexpr (CPW == 2) {
        *reinterpret_cast<uint32_t *>(p) = h[0] | (uint32_t)h[1] << 16;
        *reinterpret_cast<uint32_t *>(p + N) = l[0] | (uint32_t)l[1] << 16;
    } else {
        p[0] = __ushort_as_bfloat16(h[0]);
        p[N] = __ushort_as_bfloat16(l[0]);
    }
}

}  // namespace dmts
