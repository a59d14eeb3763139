// Message-passing layers after the first on the tensor cores (models that run
// their contractions there, C = 128 channels).
//
// With E_ij[lm,k] = f_c(r) B_k(r) Y_lm(n) of an edge (receiver i, neighbour j)
// the layer is, per receiver,
//   T_i[lm,k][c] = sum_j E_ij[lm,k] s_j[c],   A_i[lm][c] = nu sum_k W_lkc T_i[lm,k][c]:
// the neighbour sum is a dense product [C x neighbours] x [neighbours x (lm,k)]
// for tcgen05, and the radial weights are applied once per atom instead of
// once per edge.
//
// Operands are split-fp16: v 2^n = hi + lo with hi = rn_fp16, lo = rn_fp16(v 2^n - hi)
// (22 significant bits), and hi*hi + lo*hi + hi*lo is accumulated in fp32. The
// power of two n puts a row's largest element just below 2^14, so that any
// feature range fits; scaling is exact and undone on the results. Elements more
// than 2^17 below their row's largest keep fewer bits, so each channel is first
// scaled by what the weights make of it (tc_channel_scales, api.cu): the same model
// with its channels in other units, over twelve decades, has forces off by 4e-5 of
// their RMS as before; without that scale 1e-4 at eight decades and wrong at ten.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cuda_fp16.h>

#include "edge.cuh"
#include "launch.cuh"
#include "mp.cuh"
#include "ptx.cuh"
#include "tc.cuh"

namespace dmts {

namespace {

constexpr int TC_C = 128;        // channels = TMEM lanes
constexpr int TC_KR = 8;         // radial functions
constexpr int TC_E = 64;         // edges per chunk

// Exponent n of a row scale: 2^n maps values below 2 * 2^e into fp16's upper
// range; e is kept where 2^n and its inverse are normal floats.
__device__ __forceinline__ int row_exponent(unsigned max_bits) {
    return min(max((int)(max_bits >> 23) - 127, -100), 100);
}
__device__ __forceinline__ float pow2f(int n) { return __int_as_float((127 + n) << 23); }
constexpr int TC_TOP = 13;       // scaled rows lie below 2^(TC_TOP + 1)

__device__ __forceinline__ uint32_t h2u(__half2 v) { return *reinterpret_cast<uint32_t *>(&v); }

// Split pair of two values.
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    hi = h2u(h);
    lo = h2u(__floats2half2_rn(a - f.x, b - f.y));
}
// Split pair of the products a y (lo: of the unrounded product).
__device__ __forceinline__ void split2_prod(float2 a, float2 y, uint32_t &hi, uint32_t &lo) {
    const float2 v = __fmul2_rn(a, y);
    const __half2 h = __floats2half2_rn(v.x, v.y);
    const float2 f = __half22float2(h);
    const float2 r = __ffma2_rn(a, y, make_float2(-f.x, -f.y));
    hi = h2u(h);
    lo = h2u(__floats2half2_rn(r.x, r.y));
}

// Shared-memory tiles of a chunk:
//  S (neighbour features): [hi | lo][2 channel blocks][64 edges][128 bytes], 128-byte swizzle;
//  E (basis): [hi | lo][NB blocks of 16 (lm,k)][64 edges][32 bytes], 32-byte swizzle.
constexpr uint32_t S_BLK = TC_E * 128, S_PART = 2 * S_BLK, S_BYTES = 2 * S_PART;
constexpr uint32_t E_BLK = TC_E * 32;

template <int LMAX>
struct TcDims {
    static constexpr int NL = LMAX + 1, NLM = NL * NL;
    static constexpr int NK = NLM * TC_KR;                 // (lm, k) columns used
    static constexpr int NB = (NK + 15) / 16, NN = NB * 16;   // blocks of 16, padded columns
    static constexpr uint32_t e_part = NB * E_BLK, e_bytes = 2 * e_part;
};

// ---------------------------------------------------------------- front end
// A CTA's work comes in chunks of up to 64 active edges of one receiver (the
// g-th active edge of a row is slot g % 64 of chunk g / 64, whatever skin
// entries the list holds); a row without active edges is one empty chunk. One
// warp prepares them a chunk ahead of the others: it walks the rows, tests the
// candidates (96 in flight), compacts the active ones and announces the chunk.
constexpr int TC_COMPUTE = 256, TC_THREADS = TC_COMPUTE + 32;   // eight working warps and the front end
constexpr int TC_PROD = 192;                                    // threads that form products (warps 0, 1, 4-7)

struct Chunk {
    int i, n, first, last;   // receiver (-1: no more chunks), edges, first / last chunk of its row
    int e_ref;               // largest row exponent of the row's neighbours
};

struct FrontSmem {
    uint64_t full[2];              // chunk announced
    Chunk chunk[2];
    alignas(16) float4 qd[2][TC_E];   // displacement, neighbour index
    int qe[2][TC_E];                  // neighbour's row exponent
};

__device__ __forceinline__ void front_init(FrontSmem &f) {
    mbar_init(smem_u32(&f.full[0]), 1);
    mbar_init(smem_u32(&f.full[1]), 1);
}

// bar_free completes once per chunk, when nothing reads its queue any more.
// Returns false on a timeout.
__device__ __forceinline__ bool front_end(const EdgeGeom &g, const LayerIO &io, FrontSmem &f, uint32_t bar_free,
                                          int lane) {
    constexpr int U = 3;
    const int stride = gridDim.x;
    const float rc2 = g.rc * g.rc;
    auto index = [&](int wi) { return wi < g.n_atoms ? (g.order ? __ldg(g.order + wi) : wi) : -1; };
    // staged so that no load waits for another: the index two rows ahead, the replica one row ahead
    int wi = blockIdx.x;
    int i = index(wi), i1 = index(wi + stride), i2 = index(wi + 2 * stride);
    Row cur = load_row(g, wi);
    int rep1 = i1 >= 0 ? __ldg(g.atom_rep + i1) : 0;
    int jv[U], ev[U];
    float xv[U], yv[U], zv[U];
    auto load_col = [&](int first, int end) {
#pragma unroll
        for (int u = 0; u < U; ++u) jv[u] = first + 32 * u + lane < end ? __ldg(g.col + first + 32 * u + lane) : -1;
    };
    auto load_pos = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (jv[u] >= 0) {
                xv[u] = __ldg(g.x + 3 * jv[u]);
                yv[u] = __ldg(g.x + 3 * jv[u] + 1);
                zv[u] = __ldg(g.x + 3 * jv[u] + 2);
                ev[u] = __ldg(io.s_exp + jv[u]);
            }
    };
    load_col(cur.beg, cur.end);
    load_pos();
    int k = 0;   // chunks announced
    for (; i >= 0; wi += stride) {
        const AtomGeom a = wrap_inverse(cur.a);
        const int beg = cur.beg, end = cur.end;
        // the next row, and the replica and index behind it
        Row nx;
        nx.i = i1;
        nx.beg = nx.end = 0;
        if (i1 >= 0) {
            nx.beg = __ldg(g.row_ptr + i1);
            nx.end = __ldg(g.row_ptr + i1 + 1);
            nx.a.x = __ldg(g.x + 3 * i1); nx.a.y = __ldg(g.x + 3 * i1 + 1); nx.a.z = __ldg(g.x + 3 * i1 + 2);
            nx.a.bx = __ldg(g.box + 3 * rep1); nx.a.by = __ldg(g.box + 3 * rep1 + 1); nx.a.bz = __ldg(g.box + 3 * rep1 + 2);
        }
        const int rep2 = i2 >= 0 ? __ldg(g.atom_rep + i2) : 0, i3 = index(wi + 3 * stride);
        {
            int cnt = 0, first = 1, e_ref = -128;
            auto flush = [&](bool last) {
                const int b = k & 1;
                if (lane == 0) f.chunk[b] = Chunk{i, cnt, first, last ? 1 : 0, e_ref};
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&f.full[b]));
                if (last) load_col(nx.beg, nx.end);   // the next row's candidates
                if (last) load_pos();
                // the other buffer's chunk has been consumed
                if (k > 0 && !warp_wait(bar_free, (k - 1) & 1)) return false;
                ++k;
                first = 0;
                return true;
            };
            if (end - beg > 32 * U) {
                // more candidates than are in flight: the reference exponent of the whole row first
                for (int e = beg + lane; e < end; e += 32) {
                    const int j = __ldg(g.col + e);
                    if (edge_disp(a, __ldg(g.x + 3 * j), __ldg(g.x + 3 * j + 1), __ldg(g.x + 3 * j + 2)).w < rc2)
                        e_ref = max(e_ref, __ldg(io.s_exp + j));
                }
            }
            for (int base = beg; base < end; base += 32 * U) {
                if (base > beg) {
                    load_col(base, end);
                    load_pos();
                }
                float4 d[U];
                unsigned m[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    d[u] = edge_disp(a, xv[u], yv[u], zv[u]);
                    const bool act = jv[u] >= 0 && d[u].w < rc2;
                    m[u] = __ballot_sync(DMTS_FULL, act);
                    if (act) e_ref = max(e_ref, ev[u]);
                }
                if (base == beg) e_ref = __reduce_max_sync(DMTS_FULL, e_ref);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int c = __popc(m[u]);
                    const bool act = (m[u] >> lane) & 1u;
                    int pos = cnt + __popc(m[u] & ((1u << lane) - 1u));
                    const float4 v = make_float4(d[u].x, d[u].y, d[u].z, __int_as_float(jv[u]));
                    if (act && pos < TC_E) {
                        f.qd[k & 1][pos] = v;
                        f.qe[k & 1][pos] = ev[u];
                    }
                    if (cnt + c > TC_E) {   // the chunk is full and more edges follow
                        const int rest = cnt + c - TC_E;
                        cnt = TC_E;
                        if (!flush(false)) return false;
                        pos -= TC_E;
                        if (act && pos >= 0) {
                            f.qd[k & 1][pos] = v;
                            f.qe[k & 1][pos] = ev[u];
                        }
                        cnt = rest;
                    } else {
                        cnt += c;
                    }
                }
            }
            if (!flush(true)) return false;
        }
        i = i1;
        i1 = i2;
        rep1 = rep2;
        i2 = i3;
        cur = nx;
    }
    if (lane == 0) f.chunk[k & 1] = Chunk{-1, 0, 1, 1, 0};
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&f.full[k & 1]));
    return true;
}

// One edge's radial functions and harmonics, handed from the thread that
// forms them to the threads that form the products.
struct BasisBuf {
    float4 b[2][TC_E];      // f_c B_k, scaled into fp16's range
    float Y[9][TC_E];
};

// A working warp's share of a chunk's gather: rows warp, warp + 8, ... of the
// S tile, one 16-byte piece per lane and row; `rows` may exceed the chunk's
// edges (the further rows repeat the receiver's own features).
__device__ __forceinline__ void gather_share(const FrontSmem &f, uint32_t q, int rows, uint32_t sS, const __half *s16,
                                             int warp, int lane) {
    const int n = f.chunk[q & 1].n, i = f.chunk[q & 1].i;
    int j[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) j[u] = warp + 8 * u < n ? __float_as_int(f.qd[q & 1][warp + 8 * u].w) : i;
    const uint32_t dst = sS + (lane >> 3) * S_BLK + swz128(warp, lane & 7);
    const char *src = reinterpret_cast<const char *>(s16) + 16 * lane;
#pragma unroll
    for (int u = 0; u < 8; ++u)
        if (warp + 8 * u < rows) cp_async16_relaxed(dst + u * 1024, src + (size_t)j[u] * (4 * TC_C));
}

// Products of the edges' bases with the harmonics: the E tile. Thread (e, q),
// q < 3, of the six producing warps forms the eight columns (lm, k) of row e
// for lm = q, q + 3, q + 6.
template <int LMAX>
__device__ __forceinline__ void store_products(uint8_t *pE, const BasisBuf &B, int t, int n16) {
    using D = TcDims<LMAX>;
    const int e = t & (TC_E - 1), q = t / TC_E;
    if (e >= n16) return;
    const float4 b0 = B.b[0][e], b1 = B.b[1][e];
#pragma unroll
    for (int u = 0; u < (D::NLM + 2) / 3; ++u) {
        const int lm = q + 3 * u;
        if (lm >= D::NLM) break;
        const float y = B.Y[lm][e];
        const float2 yy = make_float2(y, y);
        uint4 hi, lo;
        split2_prod(make_float2(b0.x, b0.y), yy, hi.x, lo.x);
        split2_prod(make_float2(b0.z, b0.w), yy, hi.y, lo.y);
        split2_prod(make_float2(b1.x, b1.y), yy, hi.z, lo.z);
        split2_prod(make_float2(b1.z, b1.w), yy, hi.w, lo.w);
        uint8_t *p = pE + (lm >> 1) * E_BLK + swz32(e, lm & 1);
        *reinterpret_cast<uint4 *>(p) = hi;
        *reinterpret_cast<uint4 *>(p + D::e_part) = lo;
    }
}

// Sums lm = LM0 .. LM1 - 1 of one channel from its TMEM lane.
template <int LM0, int LM1>
__device__ __forceinline__ void apply_weights(uint32_t t_lane, const float (*W)[TC_KR], float sc, float *A) {
#pragma unroll
    for (int lm0 = LM0; lm0 < LM1; lm0 += 3) {
        uint32_t t[3][8];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (lm0 + u < LM1) tmem_ld8_issue(t_lane + 8 * (lm0 + u), t[u]);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int lm = lm0 + u;
            if (lm >= LM1) continue;
            const float *w = W[LM0 == 0 && lm > 0 ? 1 : 0];   // l of lm: the group's first or second row
            float v0 = 0.f, v1 = 0.f;
#pragma unroll
            for (int k = 0; k < TC_KR; k += 2) {
                v0 = fmaf(w[k], __uint_as_float(t[u][k]), v0);
                v1 = fmaf(w[k + 1], __uint_as_float(t[u][k + 1]), v1);
            }
            A[lm - LM0] = sc * (v0 + v1);
        }
    }
}

// ------------------------------------------------------------------ forward
struct FwdTcSmem {
    uint64_t bar, basis_full[2], rest;   // MMAs done, basis formed, warps 2 and 3 done with TMEM and their gather
    uint32_t tmem;
    FrontSmem front;
    BasisBuf basis[2];
};
template <int LMAX>
constexpr size_t fwd_tc_tiles() { return S_BYTES + TcDims<LMAX>::e_bytes + 1024; }   // + alignment slack

// One CTA (three per SM), a chunk at a time. Six of the eight working warps
// form the products, then one of them starts the MMAs (into the TMEM
// accumulator D[c][(lm,k)]); warps 2 and 3 meanwhile form the next chunk's
// radial functions and harmonics (a thread per edge). When the MMAs are done
// all start the next chunk's gather and, as two groups of a thread per channel,
// apply the radial weights of their channel to l <= 1 and l = 2 (the
// receiver's last chunk). Bound by the latency of a chunk's phases (about 6,000
// cycles, of which the MMAs, limited by shared-memory reads of their operands,
// take 750); 23,558 atoms, l_max = 2: 163 us, where the same sum with the
// radial products formed per edge (on the tensor cores) took 254 us. Every mbarrier wait is bounded: on timeout the CTA
// records DMTS_E_TIMEOUT, waits (bounded) for the MMAs it issued, frees its
// tensor memory and returns.
template <int LMAX>
__global__ void __launch_bounds__(TC_THREADS, 3) k_mp_fwd_tc(EdgeGeom g, LayerIO io, float escale, int *err) {
    dep_entry(g.n_atoms <= (int)gridDim.x);
    using D = TcDims<LMAX>;
    constexpr int NL = D::NL, NLM = D::NLM, C = TC_C;
    constexpr int TMEM = 128;   // columns allocated; NN <= 80 used
    extern __shared__ uint8_t tc_smem[];
    __shared__ FwdTcSmem sm;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c = tid & (C - 1), grp = tid >> 7;
    const uint32_t raw = smem_u32(tc_smem), base = (raw + 1023u) & ~1023u;
    const uint32_t sS = base, sE = base + S_BYTES;
    uint8_t *pE = tc_smem + (base - raw) + S_BYTES;
    const uint32_t sbar = smem_u32(&sm.bar), rest = smem_u32(&sm.rest);
    const int err0 = *io.err;

    if (tid == 0) {
        mbar_init(sbar, 1);
        mbar_init(smem_u32(&sm.basis_full[0]), 2);
        mbar_init(smem_u32(&sm.basis_full[1]), 2);
        mbar_init(rest, 2);
        front_init(sm.front);
        mbar_init_fence();
    }
    if (warp == 0) tmem_alloc(smem_u32(&sm.tmem), TMEM);
    // columns past (l_max + 1)^2 K stay zero
    if (NLM < 2 * D::NB && tid < 2 * TC_E)
        *reinterpret_cast<uint4 *>(pE + (tid / TC_E) * D::e_part + (D::NB - 1) * E_BLK + swz32(tid % TC_E, 1)) =
            make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem, t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    bool aborted = false;
    uint32_t k = 0;   // chunks done

    if (err0) {
        // an earlier error: nothing is computed
    } else if (warp == 8) {
        aborted = !front_end(g, io, sm.front, sbar, lane);
    } else {
        auto full = [&](uint32_t q) { return warp_wait(smem_u32(&sm.front.full[q & 1]), (q >> 1) & 1); };
        // radial weights of channel c: l = 0, 1 in the first group, l = 2 in the second (l_max = 1: 0 | 1)
        float W[2][TC_KR];
#pragma unroll
        for (int q = 0; q < TC_KR; ++q) {
            const int l0 = grp == 0 ? 0 : LMAX, l1 = LMAX >= 1 ? 1 : 0;
            W[0][q] = __ldg(io.wrad + (l0 * TC_KR + q) * C + c);
            W[1][q] = __ldg(io.wrad + (l1 * TC_KR + q) * C + c);
        }
        constexpr uint32_t idesc = idesc_f16(C, D::NN, 1, 1);
        const uint64_t descA = smem_desc_sw(sS, S_BLK, 1024, 128), descB = smem_desc_sw(sE, E_BLK, 256, 32);
        const int warp_u = __shfl_sync(DMTS_FULL, warp, 0);
        const bool is_basis = warp == 2 || warp == 3;
        // the basis of chunk q: threads 64 .. 127, one edge each
        auto basis = [&](uint32_t q) {
            const Chunk &ch = sm.front.chunk[q & 1];
            BasisBuf &B = sm.basis[q & 1];
            const int e = tid - 64, n = ch.n;
            if (e < ((n + 15) & ~15)) {
                float b[TC_KR], Y[NLM];
#pragma unroll
                for (int u = 0; u < TC_KR; ++u) b[u] = 0.f;
#pragma unroll
                for (int u = 0; u < NLM; ++u) Y[u] = 0.f;
                if (e < n) {
                    const float4 d = sm.front.qd[q & 1][e];
                    const float r = sqrtf(d.x * d.x + d.y * d.y + d.z * d.z), inv = 1.f / r;
                    float du;
                    // the neighbour's row scale relative to the receiver's reference
                    const float fc =
                        envelope(r * g.inv_rc, g.p, &du) * escale * pow2f(max(sm.front.qe[q & 1][e] - ch.e_ref, -120));
                    bessel<TC_KR, false>(r, g.inv_rc, g.bnorm, b, nullptr);
#pragma unroll
                    for (int u = 0; u < TC_KR; ++u) b[u] *= fc;
                    sph<LMAX>(d.x * inv, d.y * inv, d.z * inv, Y);
                }
                B.b[0][e] = make_float4(b[0], b[1], b[2], b[3]);
                B.b[1][e] = make_float4(b[4], b[5], b[6], b[7]);
#pragma unroll
                for (int u = 0; u < NLM; ++u) B.Y[u][e] = Y[u];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sm.basis_full[q & 1]));
        };
        // (the rows that pad the last group of 16 are filled too: 0 x row has to stay 0)
        auto gather = [&](uint32_t q) {
            const Chunk &ch = sm.front.chunk[q & 1];
            if (ch.i >= 0) gather_share(sm.front, q, (ch.n + 15) & ~15, sS, io.s16, warp, lane);
        };
        bool ok = full(0);
        if (ok) gather(0);
        if (ok && is_basis) basis(0);
        for (;; ++k) {
            const Chunk ch = sm.front.chunk[k & 1];
            if (ok && ch.i < 0) break;
            const int n16 = (ch.n + 15) & ~15;
            if (is_basis) {
                // this warp's share of the gather has landed and its reads of
                // TMEM are done: the chunk's MMAs may start
                cp_async_wait_all();
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(rest);
                ok = full(k + 1) && ok;
                if (ok) basis(k + 1);
            } else {
                ok = warp_wait(smem_u32(&sm.basis_full[k & 1]), (k >> 1) & 1) && ok;
                if (ok) store_products<LMAX>(pE, sm.basis[k & 1], (warp < 2 ? warp : warp - 2) * 32 + lane, n16);
                cp_async_wait_all();
                fence_proxy_async_smem();
                tc_fence_before();   // the last receiver's TMEM reads
                if (!bar_sync_and(1, TC_PROD, ok)) {
                    aborted = true;
                    break;
                }
                if (warp_u == 0) {
                    ok = warp_wait(rest, k & 1);
                    tc_fence_after();
                    if (ok && elect_one()) {
                        uint64_t ad = descA, bd = descB;
                        uint32_t acc = !ch.first;
#pragma unroll 1
                        for (int ks = 0; ks < n16; ks += 16, ad += 2048 >> 4, bd += 512 >> 4) {
                            mma_f16kind(tmem, ad, bd, idesc, acc);
                            mma_f16kind(tmem, ad + (S_PART >> 4), bd, idesc, 1u);
                            mma_f16kind(tmem, ad, bd + (D::e_part >> 4), idesc, 1u);
                            acc = 1u;
                        }
                        mma_commit(sbar);
                    }
                    __syncwarp();
                }
                ok = full(k + 1) && ok;
            }
            ok = warp_wait(sbar, k & 1) && ok;
            if (!ok) {
                if (!is_basis) continue;   // to the barrier of the producing warps
                aborted = true;
                break;
            }
            gather(k + 1);
            if (!ch.last) continue;
            tc_fence_after();
            // ---- thread (group, c): A[lm][c] = nu sum_k W_lkc T[lm,k][c]
            const float sc = io.nu * pow2f(max(ch.e_ref, -100) - TC_TOP) / escale;
            constexpr int M0 = LMAX == 2 ? 4 : 1;        // lm of the first group
            float A[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            if (ch.n > 0) {   // (an empty chunk is the only one of its row)
                if (grp == 0) apply_weights<0, M0>(t_lane, W, sc, A);
                else if (LMAX >= 1) apply_weights<M0, (LMAX >= 1 ? NLM : M0)>(t_lane, W, sc, A);
            }
            const int i = ch.i;
            auto put_q = [&](int l, float v) {
                if (io.q) io.q[(size_t)i * NL * C + l * C + c] = v;
                if (io.q_bf16) st_split(io.q_bf16, i, NL * C, l * C + c, v);
            };
            float *Ai = io.A + (size_t)i * NLM * C + c;
            if (grp == 0) {
#pragma unroll
                for (int lm = 0; lm < M0; ++lm) Ai[lm * C] = A[lm];
                put_q(0, A[0] * A[0]);
                if (LMAX == 2) put_q(1, fmaf(A[3], A[3], fmaf(A[2], A[2], A[1] * A[1])));
            } else if (LMAX >= 1) {
                float v = 0.f;
#pragma unroll
                for (int lm = M0; lm < NLM; ++lm) {
                    Ai[lm * C] = A[lm - M0];
                    v = fmaf(A[lm - M0], A[lm - M0], v);
                }
                put_q(LMAX, v);
            }
        }
    }

    if (aborted && lane == 0) {
        set_error(err, DMTS_E_TIMEOUT);
        if (warp < 8) mbar_wait(sbar, k & 1);   // the MMAs issued must complete before TMEM is freed
    }
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM);
    }
}

// ------------------------------------------------------- feature split
// Warp per atom: the channels times their scale (a power of two), the row's
// largest magnitude -> exponent e, hi / lo of s 2^(TC_TOP - e).
__global__ void __launch_bounds__(256) k_feature_split(int n, const float *__restrict__ s,
                                                       const float *__restrict__ ch_scale, __half *__restrict__ s16,
                                                       int *__restrict__ s_exp) {
    dep_entry();
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;
    const float4 sc = __ldg(reinterpret_cast<const float4 *>(ch_scale) + lane);
    float4 v = __ldg(reinterpret_cast<const float4 *>(s + (size_t)i * TC_C) + lane);
    v = make_float4(v.x * sc.x, v.y * sc.y, v.z * sc.z, v.w * sc.w);
    const unsigned m = max(max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))),
                           max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w))));
    const int e = row_exponent(__reduce_max_sync(DMTS_FULL, m));
    const float f = pow2f(TC_TOP - e);
    uint2 hi, lo;
    split2(v.x * f, v.y * f, hi.x, lo.x);
    split2(v.z * f, v.w * f, hi.y, lo.y);
    uint2 *row = reinterpret_cast<uint2 *>(s16 + (size_t)i * 2 * TC_C);
    row[lane] = hi;
    row[32 + lane] = lo;
    if (lane == 0) s_exp[i] = e;
}

// Power of two that puts the basis f_c B_k Y_lm (bounded by
// 2.24 sqrt(2 / rc) K pi / rc) below 2^TC_TOP.
float basis_scale(const EdgeGeom &g) {
    const float bound = 2.24f * g.bnorm * TC_KR * 3.1415927f * g.inv_rc;
    return std::ldexp(1.f, TC_TOP - 1 - std::ilogb(bound));
}

// CTAs to launch: as many as fit on the current device at once, and TMEM's
// 512 columns per SM.
int persistent_grid(const void *fn, int threads, size_t smem, int tmem_cols) {
    return sm_count() * std::max(1, std::min(resident_ctas(fn, threads, smem, current_device()), 512 / tmem_cols));
}

template <int LMAX>
void fwd_tc_launch(const EdgeGeom &g, const LayerIO &io, int *err, cudaStream_t st) {
    constexpr size_t smem = fwd_tc_tiles<LMAX>();
    cudaFuncSetAttribute(k_mp_fwd_tc<LMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_mp_fwd_tc<LMAX>, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
    const int grid = std::min(g.n_atoms, persistent_grid(reinterpret_cast<const void *>(k_mp_fwd_tc<LMAX>), TC_THREADS, smem, 128));
    launch_dep_if(g.n_atoms <= grid, k_mp_fwd_tc<LMAX>, grid, TC_THREADS, smem, st, g, io, basis_scale(g), err);
    count_launch();
}

}  // namespace

int resident_ctas(const void *fn, int threads, size_t dyn_smem, int dev) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) return 1;
    int regs_sm = 0, smem_sm = 0, smem_blk_reserved = 0, max_thr = 0, max_blk = 0;
    cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&smem_blk_reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    cudaDeviceGetAttribute(&max_thr, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
    cudaDeviceGetAttribute(&max_blk, cudaDevAttrMaxBlocksPerMultiprocessor, dev);
    const int regs_blk = ((fa.numRegs * 32 + 255) / 256 * 256) * ((threads + 31) / 32);
    const size_t smem_blk = fa.sharedSizeBytes + dyn_smem + smem_blk_reserved;
    int n = max_blk;
    if (regs_blk > 0) n = std::min(n, regs_sm / regs_blk);
    if (smem_blk > 0) n = std::min(n, (int)(smem_sm / smem_blk));
    n = std::min(n, max_thr / threads);
    return std::max(n, 1);
}

bool mp_tc_supported(int C, int K) { return C == TC_C && K == TC_KR; }

void launch_feature_split(int n, const float *s, const float *ch_scale, void *s16, int *s_exp, cudaStream_t st) {
    if (n == 0) return;
    launch_dep(k_feature_split, (n + 7) / 8, 256, 0, st, n, s, ch_scale, static_cast<__half *>(s16), s_exp);
    count_launch();
}

void launch_mp_fwd_tc(int lmax, const EdgeGeom &g, const LayerIO &io, int *err, cudaStream_t st) {
    if (g.n_atoms == 0) return;
    if (lmax == 0) fwd_tc_launch<0>(g, io, err, st);
    else if (lmax == 1) fwd_tc_launch<1>(g, io, err, st);
    else fwd_tc_launch<2>(g, io, err, st);
}

}  // namespace dmts
