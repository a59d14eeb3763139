// fp32 contractions on the tensor cores: Out[M][N] = Act[M][K] x op(W), the
// same call as the SIMT kernel (mp.cu).
//
// Each fp32 operand value is split, on its way into shared memory, into three
// bf16 parts h + m + l (h = rn(v), m = rn(v - h), l = rn(v - h - m): 24 bits,
// bf16 has fp32's exponent range), and the six products down to 2^-16 of the
// largest are accumulated in fp32 in tensor memory: h h in two accumulators
// of its own (every other K step each), the smaller ones in a third. After
// each chunk of 64 k the accumulators are added to fp32 registers: one chain
// over all of K lets their rounding through (message-passing force of 1,000
// waters against 64 bits 1.81e-6, per chunk 1.64e-6, SIMT fp32 1.72e-6).
//
// 23,558 rows, N = K = 128: 30 -> 22 us; K = 384: 70 -> 40; N = 384 with the
// gA epilogue (216 MB): 96 -> 61. Bound by the conversion's issue slots (45
// instructions per eight values, a third of them for the weights) and, over
// 370 tiles, the second wave. At 80 to 900 rows, where a call is a chain of
// latencies, the SIMT kernel is 2 us a call faster (a whole force call 227
// against 252 us at 80 atoms), from 2,000 rows on slower (555 against 487 at
// 3,000); one kernel serves every row count, so that an atom's bits do not
// depend on its batch.
//
// Range: values from 2^-102 on keep 24 bits (below it the last part falls among
// bf16's subnormals); a sum that is not finite is formed again in fp32.
#include <algorithm>
#include <cfloat>

#include "epilogue.cuh"
#include "launch.cuh"
#include "mp.cuh"
#include "ptx.cuh"
#include "tc.cuh"

namespace dmts {

namespace {

constexpr int GS_BM = 128, GS_KC = 64;                   // tile rows, K chunk (one 128-byte row of bf16)
constexpr uint32_t GS_A = GS_BM * 128;                   // bytes of one part's tile of Act

// Tiles of 128 x BN with ST operand buffers, TH threads.
template <int BN, int ST, int TH>
struct Gs {
    static constexpr uint32_t B = BN * 128, STAGE = 3 * (GS_A + B), SMEM = ST * STAGE + 1024;   // + alignment slack
    static constexpr int UA = GS_BM * 8 / TH, UB = (BN * 8 + TH - 1) / TH;   // 8-value units per thread
    static constexpr int CW = BN * 128 / TH;             // accumulator columns per warp
    static constexpr int TMEM = 256;                     // ST sets of three accumulators of BN columns
    static constexpr int LD = BN + 1;                    // staged output tile
    static_assert(GS_BM * LD * 4 <= STAGE, "the staged tile reuses the operand tiles");
    static_assert(3 * BN * ST <= TMEM && CW % 8 == 0, "tile");
};

__device__ __forceinline__ uint32_t bf2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}
// Three parts of eight values to row r, 16-byte piece g, of the part tiles.
__device__ __forceinline__ void store_split3(uint8_t *tile, uint32_t part, int r, int g, const float *v) {
    uint32_t p[3][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float a = v[2 * q], b = v[2 * q + 1];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            p[s][q] = bf2(a, b);
            a -= __uint_as_float(p[s][q] << 16);
            b -= __uint_as_float(p[s][q] & 0xffff0000u);
        }
    }
    const uint32_t o = swz128(r, g);
#pragma unroll
    for (int s = 0; s < 3; ++s)
        *reinterpret_cast<uint4 *>(tile + s * part + o) = make_uint4(p[s][0], p[s][1], p[s][2], p[s][3]);
}

// The sums of o (columns n0 .. of row m) that are not finite, once more in fp32
// as the SIMT kernel forms them (even and odd k apart): parts of a value past
// bf16's largest (3.39e38) or of an infinity are NaN, and parts may overflow
// where their sum does not. 32 comparisons per thread where every sum is finite.
__device__ __noinline__ void sums_again(float *o, int cols, int m, int n0, int M, int N, int K,
                                        const float *__restrict__ Act, const float *__restrict__ W, int trans) {
    if (m >= M) return;
    for (int v = 0; v < cols && n0 + v < N; ++v) {
        if (fabsf(o[v]) <= FLT_MAX) continue;
        float s[2] = {0.f, 0.f};
        for (int k = 0; k < K; ++k)
            s[k & 1] = fmaf(Act[(size_t)m * K + k], trans ? W[(size_t)(n0 + v) * K + k] : W[(size_t)k * N + n0 + v], s[k & 1]);
        o[v] = s[0] + s[1];
    }
}

}  // namespace

// With one buffer a chunk is converted when the last one's MMAs are done, and
// two CTAs share an SM; with two, while they run. Every wait is bounded: on
// timeout the CTA records DMTS_E_TIMEOUT, waits (bounded) for the MMAs it
// issued, frees its tensor memory and returns.
template <int BN, int ST, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) k_gemm_split(int M, int N, int K, const float *__restrict__ Act,
                                                                 const float *__restrict__ W, int trans, int vec, Epi e,
                                                                 int *err) {
    dep_entry();
    using D = Gs<BN, ST, TH>;
    constexpr int CW = D::CW;
    extern __shared__ uint8_t gs_smem[];
    __shared__ __align__(8) uint64_t bar_mem[ST];
    __shared__ uint32_t tmem_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * GS_BM, n0 = blockIdx.x * BN;
    const uint32_t raw = smem_u32(gs_smem), base = (raw + 1023u) & ~1023u;
    uint8_t *tiles = gs_smem + (base - raw);
    const uint32_t bar = smem_u32(bar_mem);
    float va[D::UA][8], vb[D::UB][8];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < D::UA; ++u) {
            const int q = tid + u * TH, r = m0 + (q >> 3), k = k0 + 8 * (q & 7);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 t = r < M && k + 4 * h < K
                                     ? __ldg(reinterpret_cast<const float4 *>(Act + (size_t)r * K + k + 4 * h))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                va[u][4 * h] = t.x; va[u][4 * h + 1] = t.y; va[u][4 * h + 2] = t.z; va[u][4 * h + 3] = t.w;
            }
        }
#pragma unroll
        for (int u = 0; u < D::UB; ++u) {
            const int q = tid + u * TH;
            if (BN * 8 < TH && q >= BN * 8) continue;
            if (trans) {   // W [N][K]: eight consecutive k of one row
                const int r = n0 + (q >> 3), k = k0 + 8 * (q & 7);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 t = r < N && k + 4 * h < K
                                         ? __ldg(reinterpret_cast<const float4 *>(W + (size_t)r * K + k + 4 * h))
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                    vb[u][4 * h] = t.x; vb[u][4 * h + 1] = t.y; vb[u][4 * h + 2] = t.z; vb[u][4 * h + 3] = t.w;
                }
            } else {       // W [K][N]: a column's eight rows (lanes along n)
                const int r = n0 + q % BN, k = k0 + 8 * (q / BN);
#pragma unroll
                for (int h = 0; h < 8; ++h) vb[u][h] = r < N && k + h < K ? __ldg(W + (size_t)(k + h) * N + r) : 0.f;
            }
        }
    };
    load(0);
    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < ST; ++s) mbar_init(bar + 8 * s, 1);
        mbar_init_fence();
    }
    if (warp == 0) tmem_alloc(smem_u32(&tmem_sh), D::TMEM);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    constexpr uint32_t idesc = idesc_bf16(GS_BM, BN);
    const int nk = (K + GS_KC - 1) / GS_KC;
    // the sums: rows 32 (w mod 4) .., columns CW (w / 4) .. of warp w
    float acc[CW];
#pragma unroll
    for (int v = 0; v < CW; ++v) acc[v] = 0.f;
    const uint32_t t_acc = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + CW * (warp >> 2);
    auto drain = [&](int c) {
        tc_fence_after();
        const bool two = K - c * GS_KC > 16;
        const uint32_t t = t_acc + (ST == 2 ? (c & 1) * 3 * BN : 0);
#pragma unroll
        for (int q = 0; q < CW / 8; ++q) {
            uint32_t d[3][8];
            tmem_ld8_issue(t + 8 * q, d[0]);
            if (two) tmem_ld8_issue(t + BN + 8 * q, d[1]);
            tmem_ld8_issue(t + 2 * BN + 8 * q, d[2]);
            tmem_wait_ld();
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const float h = two ? __uint_as_float(d[0][v]) + __uint_as_float(d[1][v]) : __uint_as_float(d[0][v]);
                acc[8 * q + v] += h + __uint_as_float(d[2][v]);
            }
        }
        tc_fence_before();
    };
    auto bar_of = [&](int c) { return bar + (ST == 2 ? 8 * (c & 1) : 0); };
    auto parity_of = [](int c) { return (uint32_t)(ST == 2 ? (c >> 1) & 1 : c & 1); };
    auto wait = [&](int c) { return warp_wait(bar_of(c), parity_of(c)) ? 1 : 0; };   // (drain() loads TMEM warp-wide)
    int ok = 1, issued = 0;
    for (int c = 0; c < nk; ++c) {
        if (ST == 1 && c > 0) ok &= wait(c - 1);   // the tiles' last readers are done
        const uint32_t so = (ST == 2 ? (c & 1) : 0) * D::STAGE;
        if (ok) {
            uint8_t *tA = tiles + so, *tB = tA + 3 * GS_A;
#pragma unroll
            for (int u = 0; u < D::UA; ++u) {
                const int q = tid + u * TH;
                store_split3(tA, GS_A, q >> 3, q & 7, va[u]);
            }
#pragma unroll
            for (int u = 0; u < D::UB; ++u) {
                const int q = tid + u * TH;
                if (BN * 8 < TH && q >= BN * 8) continue;
                store_split3(tB, D::B, trans ? q >> 3 : q % BN, trans ? q & 7 : q / BN, vb[u]);
            }
            if (ST == 1 && c > 0) drain(c - 1);
        }
        if (c + 1 < nk) load((c + 1) * GS_KC);
        fence_proxy_async_smem();
        if (!__syncthreads_and(ok)) break;
        if (warp == 0) {
            tc_fence_after();
            if (elect_one()) {
                const int steps = min(GS_KC, K - c * GS_KC + 15) / 16;
                const uint32_t d = tmem + (ST == 2 ? (c & 1) * 3 * BN : 0), small = d + 2 * BN;
                for (int s = 0; s < steps; ++s) {   // K steps: accumulator s % 2 of h h
                    const uint64_t a = smem_desc(base + so + 32 * s), b = smem_desc(base + so + 3 * GS_A + 32 * s);
                    constexpr uint32_t pa = GS_A >> 4, pb = D::B >> 4;
                    mma_f16kind(small, a + 2 * pa, b, idesc, s > 0);
                    mma_f16kind(small, a, b + 2 * pb, idesc, 1u);
                    mma_f16kind(small, a + pa, b + pb, idesc, 1u);
                    mma_f16kind(small, a + pa, b, idesc, 1u);
                    mma_f16kind(small, a, b + pb, idesc, 1u);
                    mma_f16kind(d + (s & 1) * BN, a, b, idesc, s > 1);
                }
                mma_commit(bar + (ST == 2 ? 8 * (c & 1) : 0));
            }
            __syncwarp();
        }
        issued = c + 1;
        if (ST == 2 && c > 0) {
            ok &= wait(c - 1);
            if (ok) drain(c - 1);
        }
    }
    if (ok) ok = wait(issued - 1);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            set_error(err, (int)DMTS_E_TIMEOUT);
            // the MMAs issued, once more
            for (int c = max(0, issued - ST); c < issued; ++c) mbar_wait(bar_of(c), parity_of(c));
        }
    } else {
        drain(nk - 1);
        float *tile = reinterpret_cast<float *>(tiles);
        float *o = tile + (32 * (warp & 3) + lane) * D::LD + CW * (warp >> 2);
#pragma unroll
        for (int v = 0; v < CW; ++v) o[v] = acc[v];
        bool finite = true;
#pragma unroll
        for (int v = 0; v < CW; ++v) finite = finite && fabsf(acc[v]) <= FLT_MAX;
        if (!finite) sums_again(o, CW, m0 + 32 * (warp & 3) + lane, n0 + CW * (warp >> 2), M, N, K, Act, W, trans);
        __syncthreads();
        const int rows = min(GS_BM, M - m0), cols = min(BN, N - n0);
        if (vec) epilogue_tile_v4(e, N, rows, m0, n0, cols, tile, D::LD);
        else epilogue_tile(e, N, rows, m0, n0, cols, tile, D::LD);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, D::TMEM);
    }
}

template <int BN, int ST, int TH, int MINB>
static void gemm_split_launch(int M, int N, int K, const float *Act, const float *W, int trans, const Epi &e, int *err,
                              cudaStream_t st) {
    constexpr uint32_t smem = Gs<BN, ST, TH>::SMEM;
    cudaFuncSetAttribute(k_gemm_split<BN, ST, TH, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    dim3 grid((N + BN - 1) / BN, (M + GS_BM - 1) / GS_BM);
    launch_dep(k_gemm_split<BN, ST, TH, MINB>, grid, TH, smem, st, M, N, K, Act, W, trans,
                                                               N % 4 == 0 && epilogue_vectorizable(e), e, err);
    count_launch();
}

void launch_gemm_split(int M, int N, int K, const float *Act, const float *W, int trans, const Epi &e, int *err,
                       cudaStream_t st) {
    if (M == 0) return;
    const int n_sm = sm_count();
    // narrow tiles, 512 threads and two buffers while they fit on the GPU at
    // once: a force call of 80 atoms 252 us against 297, of 3,000 487 against
    // 534; the products and their order are the same
    if ((long long)((M + GS_BM - 1) / GS_BM) * ((N + 31) / 32) > n_sm) gemm_split_launch<64, 1, 256, 2>(M, N, K, Act, W, trans, e, err, st);
    else gemm_split_launch<32, 2, 512, 1>(M, N, K, Act, W, trans, e, err, st);
}

}  // namespace dmts
