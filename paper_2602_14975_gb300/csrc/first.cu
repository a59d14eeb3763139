// First message-passing layer and its adjoint, factored over species.
//
// The first layer's input features are the species embedding, s_j = emb[z_j],
// so the neighbour sum separates from the channels:
//   A_i[lm][c] = nu sum_z emb[z][c] sum_k W_lkc T_i[z][lm][k],
//   T_i[z][lm][k] = sum over neighbours j of species z of f_c B_k Y_lm.
// T holds (l_max+1)^2 K numbers per species present, whatever the number of
// channels: an edge costs (l_max+1)^2 K products instead of
// (K (l_max+1) + (l_max+1)^2) C, no neighbour feature is gathered, and the
// channel sums are paid once per atom. The adjoint factors the same way: with
//   Q_i[z][lm][k] = sum_c gA_i[lm][c] W_lkc emb[z][c]
// the force on i of the directed edge i <- j is
//   f_ij = nu (rho n + sum_lm beta_lm dY_lm/dd),   z = z_j,
//   rho = sum_lm Y_lm sum_k (f_c B_k)' Q[z][lm][k],  beta_lm = sum_k f_c B_k Q[z][lm][k],
// which enters F_i with + and F_j with - in 32.32 fixed point.
//
// Bound by the latency and shared-memory wavefronts of one warp per atom (60 %
// of the L1 data pipe, 47 % of issue slots); 23,558 atoms, C = 128, l_max = 2:
// forward 300 -> 115 us and adjoint 503 -> 115 us against the general layer's
// kernels; the NC layer (C = 64, l_max = 1) 70 -> 45 us.
//
// The NC model has this layer only; the conservative model runs it once and
// the general layers (mp.cu, mp_tc.cu) after it.
#include <algorithm>

#include "edge.cuh"
#include "launch.cuh"
#include "mp.cuh"
#include "pack.cuh"

namespace dmts {

namespace {

constexpr int FL_K = 8;      // radial functions: lane = (k, g), k = lane % 8

// Active edges of the current row wait here until 32 are there; the g-th
// active edge of a row is always taken by lane g % 32 of batch g / 32, so
// that no sum depends on the skin entries a list happens to hold.
constexpr int FL_UNIT = 3;      // candidates per lane and sweep step, loaded together
constexpr int FL_QUEUE = 128;   // at most 31 + 96 wait

// Sweeps the row [beg, end): batch(n) is called with n <= 32 queued edges,
// the e-th at queue[(taken + e) % FL_QUEUE] (displacement; w: 8 j + species).
template <class Fn>
__device__ __forceinline__ void sweep_row(const EdgeGeom &g, const uint8_t *species, int n_species,
                                          const AtomGeom &a, int beg, int end, float4 *queue, int lane, Fn batch) {
    const float rc2 = g.rc * g.rc;
    int queued = 0, taken = 0;
    for (int base = beg; base < end; base += 32 * FL_UNIT) {
        int j[FL_UNIT];
        float4 d[FL_UNIT];
#pragma unroll
        for (int u = 0; u < FL_UNIT; ++u) j[u] = base + 32 * u + lane < end ? __ldg(g.col + base + 32 * u + lane) : -1;
#pragma unroll
        for (int u = 0; u < FL_UNIT; ++u) {
            d[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j[u] >= 0)
                d[u] = make_float4(__ldg(g.x + 3 * j[u]), __ldg(g.x + 3 * j[u] + 1), __ldg(g.x + 3 * j[u] + 2),
                                   __int_as_float((j[u] << 3) | min((int)__ldg(species + j[u]), n_species - 1)));
        }
#pragma unroll
        for (int u = 0; u < FL_UNIT; ++u) {
            d[u].x = min_img(d[u].x - a.x, a.bx, a.ibx);
            d[u].y = min_img(d[u].y - a.y, a.by, a.iby);
            d[u].z = min_img(d[u].z - a.z, a.bz, a.ibz);
            const bool act = j[u] >= 0 && d[u].x * d[u].x + d[u].y * d[u].y + d[u].z * d[u].z < rc2;
            const unsigned m = __ballot_sync(DMTS_FULL, act);
            if (act) queue[(queued + __popc(m & ((1u << lane) - 1u))) & (FL_QUEUE - 1)] = d[u];
            queued += __popc(m);
        }
        __syncwarp();
        const bool last = base + 32 * FL_UNIT >= end;
        while (queued - taken >= (last ? 1 : 32)) {
            const int n = min(32, queued - taken);
            batch(taken, n);
            taken += n;
        }
    }
}

// ------------------------------------------------------------------ forward
template <int C, int LMAX>
struct FirstFwdSmem {
    static constexpr int NL = LMAX + 1, NLM = NL * NL;
    // 20 warps per SM at l_max = 2 (shared memory), 24 otherwise (registers)
    static constexpr int WARPS = LMAX >= 2 ? 10 : 8, CTAS = LMAX >= 2 ? 2 : 3;
    // edge record: f_c B_k, then Y_lm as [lm % 4][lm / 4] so that lane (k, g)
    // reads its harmonics with one load; 12 and 28 floats: 16-byte stores of
    // eight records fall into distinct banks
    static constexpr int SLOTS = (NLM + 3) / 4;
    static constexpr int RS = SLOTS == 1 ? 12 : 28;
    // T of one species, every value twice (both halves of a packed operand)
    static constexpr int TS = 2 * NLM * FL_K;
    // floats: weights, embedding, tensor-head weights; per warp: queue, records, T
    static constexpr int w_f = NL * FL_K * C;
    static constexpr size_t bytes(int S) {
        const size_t cta = w_f + (size_t)S * C + 4 * (size_t)S * FL_K;   // weights, embedding, tensor-head weights
        return 4 * (cta + WARPS * (4 * FL_QUEUE + 32 * RS + (size_t)S * TS + 4));
    }
};

// A warp per atom. Per batch of 32 edges each lane
// embeds one edge and writes its record in species order; then lane (k, g)
// adds f_c B_k Y_lm over the edges of each species for lm = g, g + 4, 8 (one
// ascending chain per sum), and at the row's end the lanes own C / 32
// channels each and contract T with the weights, which the CTA keeps in
// shared memory.
template <int C, int LMAX>
__global__ void __launch_bounds__((FirstFwdSmem<C, LMAX>::WARPS * 32), (FirstFwdSmem<C, LMAX>::CTAS)) k_first_fwd(EdgeGeom g, FirstIO io) {
    dep_entry(g.n_atoms <= (int)(gridDim.x * (blockDim.x / 32)));
    using SM = FirstFwdSmem<C, LMAX>;
    constexpr int NL = SM::NL, NLM = SM::NLM, RS = SM::RS, TS = SM::TS, SLOTS = SM::SLOTS, WARPS = SM::WARPS;
    // channels in passes of 64 (two per lane): half the registers of one pass at C = 128
    constexpr int CP = C >= 64 ? 64 : C, CPW = CP / 32;
    using T = typename Pack<CPW>::T;
    constexpr int NP = Pack<CPW>::NP, PW = Pack<CPW>::W;
    extern __shared__ __align__(16) float fl_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, S = io.n_species;
    float *sW = fl_smem, *sE = sW + SM::w_f, *sUW = sE + S * C;
    float4 *queue = reinterpret_cast<float4 *>(sUW + 4 * S * FL_K) + warp * FL_QUEUE;
    float *per = reinterpret_cast<float *>(reinterpret_cast<float4 *>(sUW + 4 * S * FL_K) + WARPS * FL_QUEUE);
    float *sT = per + warp * S * TS;                       // 16-byte aligned: TS is a multiple of 8
    float *rec = per + WARPS * S * TS + warp * 32 * RS;
    const int err0 = *io.err;
    // the warp's first atom is on its way while the weights are loaded, and
    // each later one while the current one is worked on
    const int stride = gridDim.x * WARPS;
    int wi = blockIdx.x * WARPS + warp;
    Row nx = load_row(g, wi);
    for (int q = threadIdx.x; q < SM::w_f / 4; q += blockDim.x)
        reinterpret_cast<float4 *>(sW)[q] = __ldg(reinterpret_cast<const float4 *>(io.wrad) + q);
    if (LMAX >= 1 && io.V)
        for (int q = threadIdx.x; q < io.n_l * S * FL_K; q += blockDim.x) sUW[q] = __ldg(io.UW + q);
    for (int q = threadIdx.x; q < S * C; q += blockDim.x) sE[q] = __ldg(io.emb + q);
    __syncthreads();
    if (err0) return;
    const int k = lane & 7, grp = lane >> 3;
    for (; wi < g.n_atoms; wi += stride) {
        const int i = nx.i, beg = nx.beg, end = nx.end;
        const AtomGeom a = wrap_inverse(nx.a);
        for (int q = lane; q < S * TS; q += 32) sT[q] = 0.f;
        unsigned present = 0;
        __syncwarp();
        sweep_row(g, io.species, S, a, beg, end, queue, lane, [&](int taken, int n) {
            int z = -1;
            float B[FL_K], Y[NLM];
            if (lane < n) {
                const float4 d = queue[(taken + lane) & (FL_QUEUE - 1)];
                z = __float_as_int(d.w) & 7;
                const float r = sqrtf(d.x * d.x + d.y * d.y + d.z * d.z), inv = 1.f / r;
                float du;
                const float fc = envelope(r * g.inv_rc, g.p, &du);
                bessel<FL_K, false>(r, g.inv_rc, g.bnorm, B, nullptr);
#pragma unroll
                for (int q = 0; q < FL_K; ++q) B[q] *= fc;
                sph<LMAX>(d.x * inv, d.y * inv, d.z * inv, Y);
            }
            int pos = 0, base = 0;
            unsigned long long cnt = 0;                    // edges per species, eight bits each
            for (int s = 0; s < S; ++s) {
                const unsigned m = __ballot_sync(DMTS_FULL, z == s);
                if (z == s) pos = base + __popc(m & ((1u << lane) - 1u));
                base += __popc(m);
                cnt |= (unsigned long long)__popc(m) << (8 * s);
            }
            if (z >= 0) {
                float4 *r = reinterpret_cast<float4 *>(rec + pos * RS);
                r[0] = make_float4(B[0], B[1], B[2], B[3]);
                r[1] = make_float4(B[4], B[5], B[6], B[7]);
                if constexpr (SLOTS == 1) {
                    r[2] = make_float4(Y[0], NLM > 1 ? Y[1 % NLM] : 0.f, NLM > 1 ? Y[2 % NLM] : 0.f, NLM > 1 ? Y[3 % NLM] : 0.f);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) r[2 + q] = make_float4(Y[q], Y[q + 4], q == 0 ? Y[8] : 0.f, 0.f);
                }
            }
            __syncwarp();
            const float *r = rec;
            for (int s = 0; s < S; ++s) {
                const int ns = (int)(cnt >> (8 * s)) & 255;
                if (ns == 0) continue;
                present |= 1u << s;
                float2 *t = reinterpret_cast<float2 *>(sT + s * TS) + k;
                float acc[SLOTS];
#pragma unroll
                for (int q = 0; q < SLOTS; ++q) acc[q] = grp + 4 * q < NLM ? t[(grp + 4 * q) * FL_K].x : 0.f;
#pragma unroll 4
                for (int e = 0; e < ns; ++e, r += RS) {
                    const float b = r[k];
                    if constexpr (SLOTS == 1) {
                        acc[0] = fmaf(b, r[FL_K + grp], acc[0]);
                    } else {
                        const float4 y = *reinterpret_cast<const float4 *>(r + FL_K + 4 * grp);
                        acc[0] = fmaf(b, y.x, acc[0]);
                        acc[1] = fmaf(b, y.y, acc[1]);
                        acc[2] = fmaf(b, y.z, acc[2]);
                    }
                }
#pragma unroll
                for (int q = 0; q < SLOTS; ++q)
                    if (grp + 4 * q < NLM) t[(grp + 4 * q) * FL_K] = make_float2(acc[q], acc[q]);
            }
            __syncwarp();   // records and queue slots read before they are overwritten
        });
        __syncwarp();
        nx = load_row(g, wi + stride);
        if (io.T)
            for (int q = lane; q < S * NLM * FL_K; q += 32) io.T[(size_t)i * S * NLM * FL_K + q] = sT[2 * q];
        // ---- channel sums
#pragma unroll 1
        for (int c0 = lane * CPW; c0 < C; c0 += CP) {
            T A[NLM][NP];
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) A[lm][0] = vdup<T>(0.f);
            for (unsigned ms = present; ms; ms &= ms - 1) {
                const int s = __ffs(ms) - 1;
                T e[NP];
                ldp_s<CPW>(sE + s * C + c0, e);
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    T w[FL_K][NP];
#pragma unroll
                    for (int q = 0; q < FL_K; ++q) ldp_s<CPW>(sW + (l * FL_K + q) * C + c0, w[q]);
#pragma unroll
                    for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                        T u = vdup<T>(0.f);
#pragma unroll
                        for (int q = 0; q < FL_K; q += 2) {
                            const float4 t = *reinterpret_cast<const float4 *>(sT + s * TS + 2 * (lm * FL_K + q));
                            u = vfma(w[q][0], vpair<T>(t.x, t.y), u);
                            u = vfma(w[q + 1][0], vpair<T>(t.z, t.w), u);
                        }
                        A[lm][0] = vfma(e[0], u, A[lm][0]);
                    }
                }
            }
            const T nu = vdup<T>(io.nu);
            T qv[NL][NP];
#pragma unroll
            for (int l = 0; l < NL; ++l) qv[l][0] = vdup<T>(0.f);
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) {
                const int l = lm == 0 ? 0 : (lm < 4 ? 1 : 2);
                A[lm][0] = vmul(nu, A[lm][0]);
                qv[l][0] = vfma(A[lm][0], A[lm][0], qv[l][0]);
                if (io.A) stp<CPW>(io.A + ((size_t)i * NLM + lm) * C + c0, A[lm]);
            }
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                if (io.q) stp<CPW>(io.q + (size_t)i * NL * C + l * C + c0, qv[l]);
                if (io.q_bf16) st_split_p<CPW, PW>(io.q_bf16, i, NL * C, l * C + c0, qv[l]);
            }
        }
        if (LMAX >= 1 && io.V) {
            // V_h = sum_c U[h][c] A[l = 1][c] = nu sum_zk T[z][1 + a][k] UW[h][z][k]
            for (int h = 0; h < io.n_l; ++h) {
                float v = 0.f;
                for (unsigned ms = present; ms; ms &= ms - 1) {
                    const int s = __ffs(ms) - 1;
                    v = fmaf(sT[s * TS + 2 * lane], sUW[(h * S + s) * FL_K + k], v);   // T[s][lm = grp][k]
                }
                v += __shfl_xor_sync(DMTS_FULL, v, 1);
                v += __shfl_xor_sync(DMTS_FULL, v, 2);
                v += __shfl_xor_sync(DMTS_FULL, v, 4);
                if (k == 0 && grp > 0) io.V[(size_t)i * nc_v_stride(io.n_l) + 3 * h + grp - 1] = io.nu * v;
            }
        }
        __syncwarp();   // T read before the next atom clears it
    }
}

// ------------------------------------------------------------------ adjoint
template <int C, int LMAX>
struct FirstBwdSmem {
    static constexpr int NL = LMAX + 1, NLM = NL * NL, WARPS = 8;
    static constexpr int WS = C + 4;                            // weight row stride: eight rows in distinct banks
    static constexpr int QS = NLM * FL_K + 4;                   // Q of one species (rows of two species never collide)
    static constexpr size_t bytes(int S) {
        return 4 * ((size_t)NL * FL_K * WS + (size_t)S * C + WARPS * (4 * FL_QUEUE + NLM * C + (size_t)S * QS));
    }
};

// Eight warps per CTA, a warp per atom: gA_i = 2 A_i dU/dq_i in shared
// memory, then per batch of 32 edges Q for the species that are new to this
// row (lane (k, quarter) sums a quarter of the channels for its k and every
// lm, two species at a time) and one lane per edge for its force.
template <int C, int LMAX, bool VIR>
__global__ void __launch_bounds__(256, 2) k_first_bwd(EdgeGeom g, FirstIO io) {
    dep_entry(g.n_atoms <= (int)(gridDim.x * (blockDim.x / 32)));
    using SM = FirstBwdSmem<C, LMAX>;
    constexpr int NL = SM::NL, NLM = SM::NLM, CPW = C / 32, WS = SM::WS, QS = SM::QS, WARPS = SM::WARPS;
    using T = typename Pack<CPW>::T;
    constexpr int NP = Pack<CPW>::NP;
    extern __shared__ __align__(16) float fl_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, S = io.n_species;
    float *sW = fl_smem, *sE = sW + NL * FL_K * WS;
    float4 *queue = reinterpret_cast<float4 *>(sE + S * C) + warp * FL_QUEUE;
    float *per = reinterpret_cast<float *>(reinterpret_cast<float4 *>(sE + S * C) + WARPS * FL_QUEUE);
    float *sG = per + warp * NLM * C;
    float *sQ = per + WARPS * NLM * C + warp * S * QS;
    const int err0 = *io.err;
    // the warp's first atom is on its way while the weights are loaded, and
    // each later one while the current one is worked on
    const int stride = gridDim.x * WARPS;
    int wi = blockIdx.x * WARPS + warp;
    Row nx = load_row(g, wi);
    for (int q = threadIdx.x; q < NL * FL_K * C; q += blockDim.x) sW[q / C * WS + q % C] = __ldg(io.wrad + q);
    for (int q = threadIdx.x; q < S * C; q += blockDim.x) sE[q] = __ldg(io.emb + q);
    __syncthreads();
    if (err0) return;
    const int k = lane & 7, quarter = lane >> 3;
    bool bad = false;   // a term outside the fixed-point range (or not finite)
    for (; wi < g.n_atoms; wi += stride) {
        const int i = nx.i, beg = nx.beg, end = nx.end;
        const AtomGeom a = wrap_inverse(nx.a);
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            T v[NP];
            ldp<CPW>(io.gq + (size_t)i * NL * C + l * C + lane * CPW, v);
#pragma unroll
            for (int p = 0; p < NP; ++p) v[p] = vmul(vdup<T>(2.f), v[p]);
#pragma unroll
            for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                T t[NP];
                ldp<CPW>(io.A + ((size_t)i * NLM + lm) * C + lane * CPW, t);
#pragma unroll
                for (int p = 0; p < NP; ++p) t[p] = vmul(t[p], v[p]);
                stp<CPW>(sG + lm * C + lane * CPW, t);
            }
        }
        nx = load_row(g, wi + stride);
        unsigned done = 0;
        long long ox = 0, oy = 0, oz = 0, ow = 0;
        __syncwarp();
        sweep_row(g, io.species, S, a, beg, end, queue, lane, [&](int taken, int n) {
            const bool own = lane < n;
            const float4 d = queue[(taken + (own ? lane : 0)) & (FL_QUEUE - 1)];
            const int z = __float_as_int(d.w) & 7, j = __float_as_int(d.w) >> 3;
            unsigned fresh = __reduce_or_sync(DMTS_FULL, own ? 1u << z : 0u) & ~done;
            done |= fresh;
            while (fresh) {
                const int z0 = __ffs(fresh) - 1;
                fresh &= fresh - 1;
                const int z1 = fresh ? __ffs(fresh) - 1 : z0;
                fresh &= fresh - 1;
                float2 q0[NLM], q1[NLM];   // even and odd channels
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) q0[lm] = q1[lm] = make_float2(0.f, 0.f);
#pragma unroll 2
                for (int c = quarter * (C / 4); c < (quarter + 1) * (C / 4); c += 4) {
                    const float4 e0 = *reinterpret_cast<const float4 *>(sE + z0 * C + c);
                    const float4 e1 = *reinterpret_cast<const float4 *>(sE + z1 * C + c);
#pragma unroll
                    for (int l = 0; l < NL; ++l) {
                        const float4 w = *reinterpret_cast<const float4 *>(sW + (l * FL_K + k) * WS + c);
                        const float2 w0a = __fmul2_rn(make_float2(w.x, w.y), make_float2(e0.x, e0.y));
                        const float2 w0b = __fmul2_rn(make_float2(w.z, w.w), make_float2(e0.z, e0.w));
                        const float2 w1a = __fmul2_rn(make_float2(w.x, w.y), make_float2(e1.x, e1.y));
                        const float2 w1b = __fmul2_rn(make_float2(w.z, w.w), make_float2(e1.z, e1.w));
#pragma unroll
                        for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                            const float4 ga = *reinterpret_cast<const float4 *>(sG + lm * C + c);
                            const float2 ga0 = make_float2(ga.x, ga.y), ga1 = make_float2(ga.z, ga.w);
                            q0[lm] = __ffma2_rn(ga1, w0b, __ffma2_rn(ga0, w0a, q0[lm]));
                            q1[lm] = __ffma2_rn(ga1, w1b, __ffma2_rn(ga0, w1a, q1[lm]));
                        }
                    }
                }
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) {
                    // lanes (k, 0..3) hold the quarters: lanes with an even quarter keep z0, the others z1
                    float t0 = q0[lm].x + q0[lm].y, t1 = q1[lm].x + q1[lm].y;
                    const float give = (quarter & 1) ? t0 : t1;
                    float keep = (quarter & 1) ? t1 : t0;
                    keep += __shfl_xor_sync(DMTS_FULL, give, 8);
                    keep += __shfl_xor_sync(DMTS_FULL, keep, 16);
                    if (quarter < 2) sQ[(quarter ? z1 : z0) * QS + lm * FL_K + k] = keep;
                }
            }
            __syncwarp();
            if (own) {
                const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
                const float r = sqrtf(r2), inv = 1.f / r;
                float du;
                const float fc = envelope(r * g.inv_rc, g.p, &du);
                const float dfc = du * g.inv_rc;
                float B[FL_K], dB[FL_K], Y[NLM], dY[3 * NLM];
                bessel<FL_K, true>(r, g.inv_rc, g.bnorm, B, dB);
#pragma unroll
                for (int q = 0; q < FL_K; ++q) {
                    dB[q] = dfc * B[q] + fc * dB[q];
                    B[q] *= fc;
                }
                const float nx = d.x * inv, ny = d.y * inv, nz = d.z * inv;
                sph<LMAX>(nx, ny, nz, Y);
                sph_grad<LMAX>(nx, ny, nz, inv, dY);
                float rho = 0.f, px = 0.f, py = 0.f, pz = 0.f;
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) {
                    const float4 t0 = *reinterpret_cast<const float4 *>(sQ + z * QS + lm * FL_K);
                    const float4 t1 = *reinterpret_cast<const float4 *>(sQ + z * QS + lm * FL_K + 4);
                    const float tt[FL_K] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                    float sb = 0.f, sd = 0.f;
#pragma unroll
                    for (int q = 0; q < FL_K; ++q) {
                        sd = fmaf(dB[q], tt[q], sd);
                        if (lm > 0) sb = fmaf(B[q], tt[q], sb);
                    }
                    rho = fmaf(Y[lm], sd, rho);
                    if (lm > 0) {
                        px = fmaf(sb, dY[3 * lm], px);
                        py = fmaf(sb, dY[3 * lm + 1], py);
                        pz = fmaf(sb, dY[3 * lm + 2], pz);
                    }
                }
                px = io.nu * fmaf(rho, nx, px);
                py = io.nu * fmaf(rho, ny, py);
                pz = io.nu * fmaf(rho, nz, pz);
                if (fix_ok(px) && fix_ok(py) && fix_ok(pz)) {
                    const long long qx = to_fix(px), qy = to_fix(py), qz = to_fix(pz);
                    ox += qx; oy += qy; oz += qz;
                    unsigned long long *fj = io.Ffix + 3 * (size_t)j;
                    fix_add(fj, -qx);
                    fix_add(fj + 1, -qy);
                    fix_add(fj + 2, -qz);
                    if (VIR) {
                        const float wp = px * d.x + py * d.y + pz * d.z;   // dU/dd . d of this directed edge
                        if (fix_ok(wp)) ow += to_fix(wp);
                        else bad = true;
                    }
                } else {
                    bad = true;
                }
            }
            __syncwarp();   // Q and queue slots read before they are overwritten
        });
        ox = warp_sum_fix(ox);
        oy = warp_sum_fix(oy);
        oz = warp_sum_fix(oz);
        if (VIR) ow = warp_sum_fix(ow);
        if (lane == 0) {
            unsigned long long *fa = io.Ffix + 3 * (size_t)i;
            fix_add(fa, ox);
            fix_add(fa + 1, oy);
            fix_add(fa + 2, oz);
            if (VIR) fix_add(io.Wfix + i, ow);
        }
        __syncwarp();   // gA read before the next atom's is written
    }
    if (__any_sync(DMTS_FULL, bad) && lane == 0) set_error(io.err, (int)DMTS_E_NONFINITE);
}

// UW[h][z][k] = sum_c U[h][c] emb[z][c] W_1kc: one warp per value.
__global__ void k_tensor_head_weights(int C, int S, const float *emb, const float *wrad, const float *U, float *UW) {
    const int h = blockIdx.y, z = blockIdx.x, k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float t = 0.f;
    for (int c = lane; c < C; c += 32) t = fmaf(U[h * C + c] * emb[z * C + c], wrad[(FL_K + k) * C + c], t);
    t = warp_sum(t);
    if (lane == 0) UW[(h * S + z) * FL_K + k] = t;
}

// Persistent: as many CTAs as fit on the current device at once. Shared memory
// goes by the model's species, but the kernel's limit is the same whatever the
// model: it is shared by all contexts, and a smaller model's host thread must
// not lower it between another's setting and its launch.
template <class SM, class Kern>
void first_launch(Kern kern, const EdgeGeom &g, const FirstIO &io, cudaStream_t st) {
    constexpr int warps = SM::WARPS;
    constexpr size_t smem_max = SM::bytes(DMTS_MAX_SPECIES);
    static_assert(smem_max <= 227 * 1024, "shared memory of the largest model");
    const size_t smem = SM::bytes(io.n_species);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    const int fit = sm_count() * resident_ctas(reinterpret_cast<const void *>(kern), warps * 32, smem, current_device());
    const int grid = std::min((g.n_atoms + warps - 1) / warps, fit);
    launch_dep(kern, grid, warps * 32, smem, st, g, io);
    count_launch();
}

template <int C, int LMAX>
void first_fwd_c(const EdgeGeom &g, const FirstIO &io, cudaStream_t st) {
    first_launch<FirstFwdSmem<C, LMAX>>(k_first_fwd<C, LMAX>, g, io, st);
}

template <int C, int LMAX>
void first_bwd_c(const EdgeGeom &g, const FirstIO &io, cudaStream_t st) {
    if (io.Wfix) first_launch<FirstBwdSmem<C, LMAX>>(k_first_bwd<C, LMAX, true>, g, io, st);
    else first_launch<FirstBwdSmem<C, LMAX>>(k_first_bwd<C, LMAX, false>, g, io, st);
}

}  // namespace

void launch_tensor_head_weights(int C, int S, int n_l, const float *emb, const float *wrad, const float *U, float *UW,
                                cudaStream_t st) {
    k_tensor_head_weights<<<dim3(S, n_l), FL_K * 32, 0, st>>>(C, S, emb, wrad, U, UW);
    count_launch();
}

void launch_first_fwd(int C, int lmax, const EdgeGeom &g, const FirstIO &io, cudaStream_t st) {
    if (g.n_atoms == 0) return;
    DMTS_DISPATCH(first_fwd_c, C, lmax, g, io, st);
}

void launch_first_bwd(int C, int lmax, const EdgeGeom &g, const FirstIO &io, cudaStream_t st) {
    if (g.n_atoms == 0) return;
    DMTS_DISPATCH(first_bwd_c, C, lmax, g, io, st);
}

}  // namespace dmts
