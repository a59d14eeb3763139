// Fused epilogues of the node-level contractions (Epi, mp.cuh), applied to an
// output tile staged in shared memory.
#pragma once
#include "mp.cuh"

namespace dmts {

// Applies the epilogue to a rows x BN tile held in shared memory. Each
// thread takes EU elements per pass (row-major, consecutive threads on
// consecutive columns) and issues all of their global loads before any
// store, so that many loads are in flight per warp.
constexpr int EU = 4;

// Row of the residual input. The first layer's is the species embedding, read
// from the table itself: an [M][N] copy of it was a launch of its own (12 us at
// 49,152 rows of 64, 3 us at 80) and M N floats written and read.
__device__ __forceinline__ size_t res_offset(const Epi &e, int m, int N) {
    return (size_t)(e.res_row ? (int)__ldg(e.res_row + m) : m) * N;
}

__device__ __forceinline__ void epilogue_tile(const Epi &e, int N, int rows, int m0, int n0, int BN,
                                              const float *tile, int ld) {
    const int total = rows * BN;
    const int step = blockDim.x;
    for (int base = threadIdx.x; base < total; base += EU * step) {
        float v[EU];
        size_t o[EU];
        int n[EU], r_[EU];
        bool ok[EU];
#pragma unroll
        for (int u = 0; u < EU; ++u) {
            const int idx = base + u * step;
            ok[u] = idx < total;
            const int r = ok[u] ? idx / BN : 0, c = ok[u] ? idx - r * BN : 0;
            v[u] = ok[u] ? tile[r * ld + c] : 0.f;
            n[u] = n0 + c;
            r_[u] = r;
            o[u] = (size_t)(m0 + r) * N + n[u];
        }
        switch (e.mode) {
        case EPI_STORE:
#pragma unroll
            for (int u = 0; u < EU; ++u)
                if (ok[u]) {
                    e.out[o[u]] = v[u];
                    if (e.out_bf16) st_split(e.out_bf16, (size_t)(m0 + r_[u]), N, n[u], v[u]);
                }
            break;
        case EPI_BIAS_SILU: {
            float b[EU];
#pragma unroll
            for (int u = 0; u < EU; ++u) b[u] = ok[u] ? __ldg(e.bias + n[u]) : 0.f;
#pragma unroll
            for (int u = 0; u < EU; ++u)
                if (ok[u]) {
                    const float h = v[u] + b[u];
                    const float sv = silu_f(h);
                    if (e.H) e.H[o[u]] = h;
                    if (e.out) e.out[o[u]] = sv;
                    if (e.out_bf16) st_split(e.out_bf16, (size_t)(m0 + r_[u]), N, n[u], sv);
                }
            break;
        }
        case EPI_RESID: {
            float rs[EU], b[EU];
#pragma unroll
            for (int u = 0; u < EU; ++u) {
                rs[u] = ok[u] ? __ldg(e.res + res_offset(e, m0 + r_[u], N) + n[u]) : 0.f;
                b[u] = ok[u] ? __ldg(e.bias + n[u]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < EU; ++u)
                if (ok[u]) {
                    const float rr = rs[u] + v[u] + b[u];
                    e.out[o[u]] = rr;
                    if (e.out_bf16) st_split(e.out_bf16, (size_t)(m0 + r_[u]), N, n[u], rr);
                }
            break;
        }
        case EPI_DSILU: {
            float h[EU];
#pragma unroll
            for (int u = 0; u < EU; ++u) h[u] = ok[u] ? __ldg(e.H + o[u]) : 0.f;
#pragma unroll
            for (int u = 0; u < EU; ++u)
                if (ok[u]) {
                    const float rr = v[u] * dsilu_f(h[u]);
                    e.out[o[u]] = rr;
                    if (e.out_bf16) st_split(e.out_bf16, (size_t)(m0 + r_[u]), N, n[u], rr);
                }
            break;
        }
        case EPI_GA: {
            const int nlm = (e.lmax + 1) * (e.lmax + 1);
            float a[EU][5];
            size_t ib[EU];
            int l0[EU], nm[EU];
#pragma unroll
            for (int u = 0; u < EU; ++u) {
                const int l = n[u] / e.C, c = n[u] - l * e.C;
                const int m = (int)(o[u] / N);
                l0[u] = l * l;
                nm[u] = ok[u] ? 2 * l + 1 : 0;
                ib[u] = ((size_t)m * nlm + l0[u]) * e.C + c;
#pragma unroll
                for (int q = 0; q < 5; ++q) a[u][q] = q < nm[u] ? __ldg(e.A + ib[u] + (size_t)q * e.C) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < EU; ++u)
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    if (q < nm[u]) e.out[ib[u] + (size_t)q * e.C] = 2.f * a[u][q] * v[u];
            break;
        }
        case EPI_READOUT: {
            float b[EU], w[EU];
#pragma unroll
            for (int u = 0; u < EU; ++u) {
                b[u] = ok[u] ? __ldg(e.bias + n[u]) : 0.f;
                w[u] = ok[u] ? __ldg(e.wo + n[u]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < EU; ++u)
                if (ok[u]) {
                    const float z = v[u] + b[u];
                    e.out[o[u]] = w[u] * silu_f(z);
                    const float gz = e.scale * w[u] * dsilu_f(z);
                    e.out2[o[u]] = gz;
                    if (e.out_bf16) st_split(e.out_bf16, (size_t)(m0 + r_[u]), N, n[u], gz);
                }
            break;
        }
        }
    }
}

// Vector form of the epilogue, used when every array it touches is 16-byte
// aligned (bf16 copies 8-byte): each thread takes groups of four
// consecutive columns of a row, so global loads and stores are 16-byte
// vectors, and the row / column of its next group follow by additions.
__device__ __forceinline__ float4 ld4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
// Four consecutive columns of a split-bf16 copy (common.cuh): the hi parts
// at p, the lo parts at p + N (N = the logical row length).
__device__ __forceinline__ void st4_split(__nv_bfloat16 *p, int N, float4 v) {
    __nv_bfloat16 h[4], l[4];
    split_bf16(v.x, h[0], l[0]);
    split_bf16(v.y, h[1], l[1]);
    split_bf16(v.z, h[2], l[2]);
    split_bf16(v.w, h[3], l[3]);
    uint2 uh, ul;
    uh.x = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
    uh.y = (uint32_t)__bfloat16_as_ushort(h[2]) | ((uint32_t)__bfloat16_as_ushort(h[3]) << 16);
    ul.x = (uint32_t)__bfloat16_as_ushort(l[0]) | ((uint32_t)__bfloat16_as_ushort(l[1]) << 16);
    ul.y = (uint32_t)__bfloat16_as_ushort(l[2]) | ((uint32_t)__bfloat16_as_ushort(l[3]) << 16);
    *reinterpret_cast<uint2 *>(p) = uh;
    *reinterpret_cast<uint2 *>(p + N) = ul;
}
__device__ __forceinline__ float4 bias4(const float *b, int n) {
    return make_float4(__ldg(b + n), __ldg(b + n + 1), __ldg(b + n + 2), __ldg(b + n + 3));
}
__device__ __forceinline__ float4 silu4(float4 h) { return make_float4(silu_f(h.x), silu_f(h.y), silu_f(h.z), silu_f(h.w)); }

constexpr int EU4 = 2;   // groups per thread and pass

__device__ __forceinline__ void epilogue_tile_v4(const Epi &e, int N, int rows, int m0, int n0, int BN,
                                                 const float *tile, int ld) {
    const int G = BN / 4, total = rows * G, step = blockDim.x;
    const int dr = step / G, dc = step - dr * G;
    int r = threadIdx.x / G, c = threadIdx.x - (threadIdx.x / G) * G;
    const int nlm = (e.lmax + 1) * (e.lmax + 1);
    for (int base = threadIdx.x; base < total; base += EU4 * step) {
        float4 v[EU4];
        int rr[EU4], cc[EU4];
        bool ok[EU4];
#pragma unroll
        for (int u = 0; u < EU4; ++u) {
            ok[u] = base + u * step < total;
            rr[u] = r;
            cc[u] = c;
            const float *t = tile + r * ld + 4 * c;
            v[u] = ok[u] ? make_float4(t[0], t[1], t[2], t[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
            r += dr;
            c += dc;
            if (c >= G) { c -= G; ++r; }
        }
        switch (e.mode) {
        case EPI_STORE:
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                if (ok[u]) {
                    const size_t o = (size_t)(m0 + rr[u]) * N + n0 + 4 * cc[u];
                    st4(e.out + o, v[u]);
                    if (e.out_bf16) st4_split(e.out_bf16 + (size_t)(m0 + rr[u]) * 2 * N + n0 + 4 * cc[u], N, v[u]);
                }
            break;
        case EPI_BIAS_SILU:
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                if (ok[u]) {
                    const int n = n0 + 4 * cc[u];
                    const size_t o = (size_t)(m0 + rr[u]) * N + n;
                    const float4 b = bias4(e.bias, n);
                    const float4 h = make_float4(v[u].x + b.x, v[u].y + b.y, v[u].z + b.z, v[u].w + b.w);
                    const float4 sv = silu4(h);
                    if (e.H) st4(e.H + o, h);
                    if (e.out) st4(e.out + o, sv);
                    if (e.out_bf16) st4_split(e.out_bf16 + (size_t)(m0 + rr[u]) * 2 * N + n0 + 4 * cc[u], N, sv);
                }
            break;
        case EPI_RESID: {
            float4 rs[EU4];
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                rs[u] = ok[u] ? ld4(e.res + res_offset(e, m0 + rr[u], N) + n0 + 4 * cc[u]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                if (ok[u]) {
                    const int n = n0 + 4 * cc[u];
                    const size_t o = (size_t)(m0 + rr[u]) * N + n;
                    const float4 b = bias4(e.bias, n);
                    const float4 o4 = make_float4(rs[u].x + v[u].x + b.x, rs[u].y + v[u].y + b.y,
                                                  rs[u].z + v[u].z + b.z, rs[u].w + v[u].w + b.w);
                    st4(e.out + o, o4);
                    if (e.out_bf16) st4_split(e.out_bf16 + (size_t)(m0 + rr[u]) * 2 * N + n0 + 4 * cc[u], N, o4);
                }
            break;
        }
        case EPI_DSILU: {
            float4 h[EU4];
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                h[u] = ok[u] ? ld4(e.H + (size_t)(m0 + rr[u]) * N + n0 + 4 * cc[u]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                if (ok[u]) {
                    const size_t o = (size_t)(m0 + rr[u]) * N + n0 + 4 * cc[u];
                    const float4 o4 = make_float4(v[u].x * dsilu_f(h[u].x), v[u].y * dsilu_f(h[u].y),
                                                  v[u].z * dsilu_f(h[u].z), v[u].w * dsilu_f(h[u].w));
                    st4(e.out + o, o4);
                    if (e.out_bf16) st4_split(e.out_bf16 + (size_t)(m0 + rr[u]) * 2 * N + n0 + 4 * cc[u], N, o4);
                }
            break;
        }
        case EPI_GA: {
            // n = l C + c: the four columns share l (C % 4 == 0)
            float4 a[EU4][5];
            size_t ib[EU4];
            int nm[EU4];
#pragma unroll
            for (int u = 0; u < EU4; ++u) {
                const int n = n0 + 4 * cc[u];
                const int l = n / e.C, cch = n - l * e.C;
                nm[u] = ok[u] ? 2 * l + 1 : 0;
                ib[u] = ((size_t)(m0 + rr[u]) * nlm + l * l) * e.C + cch;
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    a[u][q] = q < nm[u] ? ld4(e.A + ib[u] + (size_t)q * e.C) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < EU4; ++u)
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    if (q < nm[u])
                        st4(e.out + ib[u] + (size_t)q * e.C,
                            make_float4(2.f * a[u][q].x * v[u].x, 2.f * a[u][q].y * v[u].y, 2.f * a[u][q].z * v[u].z,
                                        2.f * a[u][q].w * v[u].w));
            break;
        }
        case EPI_READOUT:
#pragma unroll
            for (int u = 0; u < EU4; ++u)
                if (ok[u]) {
                    const int n = n0 + 4 * cc[u];
                    const size_t o = (size_t)(m0 + rr[u]) * N + n;
                    const float4 b = bias4(e.bias, n), w = bias4(e.wo, n);
                    const float4 z = make_float4(v[u].x + b.x, v[u].y + b.y, v[u].z + b.z, v[u].w + b.w);
                    st4(e.out + o, make_float4(w.x * silu_f(z.x), w.y * silu_f(z.y), w.z * silu_f(z.z), w.w * silu_f(z.w)));
                    const float4 gz = make_float4(e.scale * w.x * dsilu_f(z.x), e.scale * w.y * dsilu_f(z.y),
                                                  e.scale * w.z * dsilu_f(z.z), e.scale * w.w * dsilu_f(z.w));
                    st4(e.out2 + o, gz);
                    if (e.out_bf16) st4_split(e.out_bf16 + (size_t)(m0 + rr[u]) * 2 * N + n0 + 4 * cc[u], N, gz);
                }
            break;
        }
    }
}

// Whether the vector form may be used: every array 16-byte aligned (bf16
// copies 8-byte), channels in groups of four.
inline int epilogue_vectorizable(const Epi &e) {
    auto al = [](const void *p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; };
    return al(e.out, 16) && al(e.out2, 16) && al(e.H, 16) && al(e.res, 16) && al(e.A, 16) && al(e.out_bf16, 8) &&
           (e.mode != EPI_GA || e.C % 4 == 0);
}

}  // namespace dmts
