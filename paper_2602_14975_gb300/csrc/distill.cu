// Adjoint of the fast force with respect to the NC model's weights
// (distillation of the NC model, Sec. 2 "Model training"): the head, the
// weight contractions, the layer's radial and tensor-head weights.
#include <algorithm>

#include "edge.cuh"
#include "md.cuh"
#include "mp.cuh"
#include "ptx.cuh"

namespace dmts {

// ------------------------------------------------- NC head adjoint (q/k)
// With F_aj = f_c S_aj (n + T_aj), S_aj = sum_{h<K} c_ajh B_h,
// T_aj = sum_t c_aj(K+t) V_at, F_ja = f_c S_ja (-n + T_ja) and
// F_a = scale sum_j (F_aj - F_ja) (+ terms without q/k), each directed pair
// enters F_a with + and F_j with -, so u = scale (gF_a - gF_j) and
//   dL/dc_ajh = f_c B_h u.(n + T_aj)   (h < K),  f_c S_aj u.V_at  (h = K + t),
//   dL/dc_jah = -f_c B_h u.(-n + T_ja) (h < K), -f_c S_ja u.V_jt  (h = K + t).
// Each pair is visited from both ends, so every atom gathers its own rows'
// gradients: no atomics, deterministic. A warp per atom; its active neighbours
// are taken 16 at a time: two lanes per edge (half of the heads each) form the
// products c and the gradients dL/dc from the neighbour's q/k row, staged in
// shared memory by bulk copies, and then lane (role, head) adds dL/dc times the
// neighbour's row over the batch's edges. Bound by issue (the row sums) and
// the rows' gather from L2. (49,152 atoms of water, 26 neighbours each: 187 us;
// a lane per head with every edge's radial part on all lanes took 669 us.)
constexpr int HB_WARPS = 4, HB_BATCH = 16;

template <int K, int NC, int NL>
struct HeadBwdSmem {
    static constexpr int H = K + NL, QKW = 2 * H * NC;
    static constexpr int RSTR = QKW + 4;       // padded row stride: conflict-free 16-byte reads
    static constexpr int GSTR = 2 * H + 1;
    static constexpr int HH = (H + 1) / 2;     // heads per lane of a pair; the tensor heads are the second lane's
    static_assert(HH <= K && 2 * H <= 32, "head split");
    alignas(16) float rows[HB_BATCH * RSTR];
    alignas(16) float own[QKW];
    float grad[HB_BATCH * GSTR];
    float va[3 * NL];
    float4 queue[64];                          // displacement, neighbour index
    uint64_t bar;
};

template <int K, int NC, int NL>
__global__ void __launch_bounds__(HB_WARPS * 32) k_nc_head_bwd(NCHeadArgs g, const float *__restrict__ gF,
                                                               float *__restrict__ gQK, float *__restrict__ gV) {
    using SM = HeadBwdSmem<K, NC, NL>;
    constexpr int H = SM::H, QKW = SM::QKW, RSTR = SM::RSTR, GSTR = SM::GSTR, HH = SM::HH, VS = nc_v_stride(NL);
    extern __shared__ __align__(16) unsigned char hb_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    SM &sm = reinterpret_cast<SM *>(hb_smem)[warp];
    const int wa = blockIdx.x * HB_WARPS + warp;
    if (wa >= g.n_atoms || *g.err) return;
    const uint32_t bar = smem_u32(&sm.bar);
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
    }
    const int a = g.order ? __ldg(g.order + wa) : wa;
    const int beg = g.row_ptr[a], end = g.row_ptr[a + 1];
    AtomGeom ge;
    const int rep = g.atom_rep[a];
    ge.bx = g.box[3 * rep]; ge.by = g.box[3 * rep + 1]; ge.bz = g.box[3 * rep + 2];
    ge.x = g.x[3 * a]; ge.y = g.x[3 * a + 1]; ge.z = g.x[3 * a + 2];
    ge = wrap_inverse(ge);
    for (int q = lane; q < QKW / 4; q += 32)
        reinterpret_cast<float4 *>(sm.own)[q] = __ldg(reinterpret_cast<const float4 *>(g.QK + (size_t)a * QKW) + q);
    if (lane < 3 * NL) sm.va[lane] = __ldg(g.V + (size_t)a * VS + lane);
    const float gax = gF[3 * a], gay = gF[3 * a + 1], gaz = gF[3 * a + 2];
    const float rc2 = g.rc * g.rc, isnc = rsqrtf((float)NC);
    const int slot = lane & (HB_BATCH - 1), half = lane / HB_BATCH;
    float acc[NC], accv[NL][3];
#pragma unroll
    for (int d = 0; d < NC; ++d) acc[d] = 0.f;
#pragma unroll
    for (int t = 0; t < NL; ++t) accv[t][0] = accv[t][1] = accv[t][2] = 0.f;
    uint32_t phase = 0;
    __syncwarp();

    auto batch = [&](int taken, int nb) -> bool {
        const float4 e = sm.queue[(taken + (slot < nb ? slot : 0)) & 63];
        const int j = __float_as_int(e.w);
        const bool live = slot < nb;
        fence_proxy_async_smem();   // earlier reads of the rows before the copies overwrite them
        if (lane == 0) mbar_expect_tx(bar, (uint32_t)nb * QKW * 4);
        __syncwarp();
        if (live && half == 0) bulk_g2s(smem_u32(sm.rows + slot * RSTR), g.QK + (size_t)j * QKW, QKW * 4, bar);
        float vj[3 * NL];
#pragma unroll
        for (int q = 0; q < 3 * NL; ++q) vj[q] = half == 1 ? __ldg(g.V + (size_t)j * VS + q) : 0.f;
        const float ux = g.scale * (gax - __ldg(gF + 3 * j)), uy = g.scale * (gay - __ldg(gF + 3 * j + 1)),
                    uz = g.scale * (gaz - __ldg(gF + 3 * j + 2));
        const float r = sqrtf(e.x * e.x + e.y * e.y + e.z * e.z), inv = 1.f / r;
        float du;
        const float fc = live ? envelope(r * g.inv_rc, g.p, &du) : 0.f;
        float B[K], Bh[HH];
        bessel<K, false>(r, g.inv_rc, g.bnorm, B, nullptr);
#pragma unroll
        for (int hl = 0; hl < HH; ++hl)
            Bh[hl] = half == 0 ? B[hl] : (HH + hl < K ? B[HH + hl < K ? HH + hl : 0] : 0.f);
        if (!__all_sync(DMTS_FULL, mbar_wait(bar, phase))) {
            if (lane == 0) atomicCAS(g.err, 0, (int)DMTS_E_TIMEOUT);
            mbar_wait(bar, phase);   // the copies in flight, once more
            return false;
        }
        phase ^= 1u;
        // this lane's heads h = half * HH + hl: c_aj, c_ja and their sums S, T
        float caj[HH], cja[HH], part[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // Saj, Sja, Taj (3), Tja (3)
        const float *row = sm.rows + slot * RSTR;
#pragma unroll
        for (int hl = 0; hl < HH; ++hl) {
            const int h = half * HH + hl;
            caj[hl] = cja[hl] = 0.f;
            if (h < H && live) {
#pragma unroll
                for (int q = 0; q < NC / 4; ++q) {
                    const float4 qj = *reinterpret_cast<const float4 *>(row + h * NC + 4 * q);
                    const float4 kj = *reinterpret_cast<const float4 *>(row + (H + h) * NC + 4 * q);
                    const float4 qi = *reinterpret_cast<const float4 *>(sm.own + h * NC + 4 * q);
                    const float4 ki = *reinterpret_cast<const float4 *>(sm.own + (H + h) * NC + 4 * q);
                    caj[hl] = fmaf(qi.x, kj.x, fmaf(qi.y, kj.y, fmaf(qi.z, kj.z, fmaf(qi.w, kj.w, caj[hl]))));
                    cja[hl] = fmaf(qj.x, ki.x, fmaf(qj.y, ki.y, fmaf(qj.z, ki.z, fmaf(qj.w, ki.w, cja[hl]))));
                }
                caj[hl] *= isnc;
                cja[hl] *= isnc;
                if (h < K) {
                    part[0] = fmaf(caj[hl], Bh[hl], part[0]);
                    part[1] = fmaf(cja[hl], Bh[hl], part[1]);
                } else {
                    const int t = HH + hl - K;   // (the second lane's heads: t is static)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        part[2 + q] = fmaf(caj[hl], sm.va[3 * t + q], part[2 + q]);
                        part[5 + q] = fmaf(cja[hl], vj[3 * t + q], part[5 + q]);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) part[q] += __shfl_xor_sync(DMTS_FULL, part[q], HB_BATCH);
        const float nx = e.x * inv, ny = e.y * inv, nz = e.z * inv;
        const float paj = fc * (ux * (nx + part[2]) + uy * (ny + part[3]) + uz * (nz + part[4]));
        const float pja = -fc * (ux * (-nx + part[5]) + uy * (-ny + part[6]) + uz * (-nz + part[7]));
        const float saj = fc * part[0], sja = -fc * part[1];
#pragma unroll
        for (int hl = 0; hl < HH; ++hl) {
            const int h = half * HH + hl;
            if (h >= H) continue;
            float ga, gj;
            if (h < K) {
                ga = Bh[hl] * paj;
                gj = Bh[hl] * pja;
            } else {
                const int t = HH + hl - K;
                ga = saj * (ux * sm.va[3 * t] + uy * sm.va[3 * t + 1] + uz * sm.va[3 * t + 2]);
                gj = sja * (ux * vj[3 * t] + uy * vj[3 * t + 1] + uz * vj[3 * t + 2]);
                // V_at enters F_aj = f_c S_aj (n + sum_t c_aj(K+t) V_at) only
                const float f = saj * caj[hl];
                accv[t][0] = fmaf(f, ux, accv[t][0]);
                accv[t][1] = fmaf(f, uy, accv[t][1]);
                accv[t][2] = fmaf(f, uz, accv[t][2]);
            }
            sm.grad[slot * GSTR + h] = isnc * ga;
            sm.grad[slot * GSTR + H + h] = isnc * gj;
        }
        __syncwarp();
        // lane (role, h): dL/dq_ah = sum_j dL/dc_ajh k_jh, dL/dk_ah = sum_j dL/dc_jah q_jh
        if (lane < 2 * H) {
            const float *other = sm.rows + (lane < H ? lane + H : lane - H) * NC;
#pragma unroll 4
            for (int t = 0; t < nb; ++t) {
                const float w = sm.grad[t * GSTR + lane];
#pragma unroll
                for (int q = 0; q < NC / 4; ++q) {
                    const float4 o = *reinterpret_cast<const float4 *>(other + t * RSTR + 4 * q);
                    acc[4 * q] = fmaf(w, o.x, acc[4 * q]);
                    acc[4 * q + 1] = fmaf(w, o.y, acc[4 * q + 1]);
                    acc[4 * q + 2] = fmaf(w, o.z, acc[4 * q + 2]);
                    acc[4 * q + 3] = fmaf(w, o.w, acc[4 * q + 3]);
                }
            }
        }
        __syncwarp();
        return true;
    };

    int queued = 0, taken = 0;
    for (int base = beg; base < end; base += 32) {
        const int e = base + lane;
        bool act = false;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < end) {
            const int j = __ldg(g.col + e);
            d = edge_disp(ge, __ldg(g.x + 3 * j), __ldg(g.x + 3 * j + 1), __ldg(g.x + 3 * j + 2));
            act = d.w < rc2;
            d.w = __int_as_float(j);
        }
        const unsigned m = __ballot_sync(DMTS_FULL, act);
        if (act) sm.queue[(queued + __popc(m & ((1u << lane) - 1u))) & 63] = d;
        queued += __popc(m);
        __syncwarp();
        while (queued - taken >= HB_BATCH) {
            if (!batch(taken, HB_BATCH)) return;
            taken += HB_BATCH;
        }
    }
    if (queued > taken && !batch(taken, queued - taken)) return;
    if (gV) {
#pragma unroll
        for (int t = 0; t < NL; ++t)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float v = warp_sum(accv[t][q]);
                if (lane == 0) gV[((size_t)a * NL + t) * 3 + q] = v;
            }
    }
    if (lane < 2 * H) {
        float4 *o = reinterpret_cast<float4 *>(gQK + (size_t)a * QKW + lane * NC);
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) o[q] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    }
}

template <int K, int NC, int NL>
static void nc_head_bwd_launch(const NCHeadArgs &a, const float *gF, float *gQK, float *gV, cudaStream_t st) {
    constexpr size_t smem = HB_WARPS * sizeof(HeadBwdSmem<K, NC, NL>);
    cudaFuncSetAttribute(k_nc_head_bwd<K, NC, NL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_nc_head_bwd<K, NC, NL><<<(a.n_atoms + HB_WARPS - 1) / HB_WARPS, HB_WARPS * 32, smem, st>>>(a, gF, gQK, gV);
    count_launch();
}

void launch_nc_head_bwd(int K, int n_c, int n_l, const NCHeadArgs &a, const float *gF, float *gQK, float *gV,
                        cudaStream_t st) {
    if (a.n_atoms == 0) return;
    if (K == 8 && n_c == 8 && n_l == 2) nc_head_bwd_launch<8, 8, 2>(a, gF, gQK, gV, st);
    else if (K == 8 && n_c == 8 && n_l == 1) nc_head_bwd_launch<8, 8, 1>(a, gF, gQK, gV, st);
    else if (K == 8 && n_c == 8 && n_l == 3) nc_head_bwd_launch<8, 8, 3>(a, gF, gQK, gV, st);
    else if (K == 8 && n_c == 8 && n_l == 4) nc_head_bwd_launch<8, 8, 4>(a, gF, gQK, gV, st);
}

// ------------------------------------------------ weight gradients (A^T B)
// A block computes a 64 x 64 output tile over one slice of atoms, 4 x 4
// outputs per thread, in atom order; the next 16 atoms' rows are loaded while
// the current ones are multiplied. The slices, 256 atoms
// or more each, fill the chip: the outputs alone are 2 to 6 tiles. (49,152
// atoms, outputs 160 x 64, 64 x 64 and 64 x 128: 41, 20 and 29 us; 32 x 32 tiles
// of one output column per thread over 64 slices took 122, 86 and 103 us.)
constexpr int ATB_T = 64, ATB_CH = 16;

__global__ void __launch_bounds__(256) k_atb_part(int N, int O, int I, const float *__restrict__ G,
                                                 const float *__restrict__ X, float *__restrict__ part, int with_cs,
                                                 int slices) {
    __shared__ __align__(16) float Gs[2][ATB_CH][ATB_T], Xs[2][ATB_CH][ATB_T];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int o0 = blockIdx.x * ATB_T, i0 = blockIdx.y * ATB_T, sl = blockIdx.z;
    const int per = (N + slices - 1) / slices, a0 = min(N, sl * per), a1 = min(N, a0 + per);
    // thread (ty, tx) loads four columns of atom row ty
    const int lc = 4 * tx;
    auto load = [&](int c0, float4 &gv, float4 &xv) {
        const int at = c0 + ty;
        gv = xv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (at < a1 && o0 + lc < O) gv = __ldg(reinterpret_cast<const float4 *>(G + (size_t)at * O + o0 + lc));
        if (at < a1 && i0 + lc < I) xv = __ldg(reinterpret_cast<const float4 *>(X + (size_t)at * I + i0 + lc));
    };
    float acc[4][4] = {}, cs[4] = {0.f, 0.f, 0.f, 0.f};
    float4 gv, xv;
    load(a0, gv, xv);
    int b = 0;
    for (int c0 = a0; c0 < a1; c0 += ATB_CH, b ^= 1) {
        *reinterpret_cast<float4 *>(&Gs[b][ty][lc]) = gv;
        *reinterpret_cast<float4 *>(&Xs[b][ty][lc]) = xv;
        __syncthreads();   // (two buffers: the previous step's reads are behind its successor's barrier)
        if (c0 + ATB_CH < a1) load(c0 + ATB_CH, gv, xv);
#pragma unroll
        for (int aa = 0; aa < ATB_CH; ++aa) {
            const float4 g4 = *reinterpret_cast<const float4 *>(&Gs[b][aa][4 * ty]);
            const float4 x4 = *reinterpret_cast<const float4 *>(&Xs[b][aa][4 * tx]);
            const float gg[4] = {g4.x, g4.y, g4.z, g4.w}, xx[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int p = 0; p < 4; ++p) {
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(gg[p], xx[q], acc[p][q]);
                cs[p] += gg[p];
            }
        }
    }
    float *pp = part + (size_t)sl * O * (I + 1);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int o = o0 + 4 * ty + p;
        if (o >= O) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i0 + 4 * tx + q < I) pp[(size_t)o * (I + 1) + i0 + 4 * tx + q] = acc[p][q];
        if (with_cs && blockIdx.y == 0 && tx == 0) pp[(size_t)o * (I + 1) + I] = cs[p];
    }
}

// Sum over the slices: eight warps add every eighth slice, in order, and their
// sums are added in warp order.
__global__ void __launch_bounds__(256) k_atb_reduce(int O, int I, const float *__restrict__ part,
                                                    float *__restrict__ out, float *__restrict__ cs, int slices) {
    __shared__ float red[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * 32 + lane;
    const int o = q / (I + 1), i = q % (I + 1);
    const bool live = q < O * (I + 1) && (i < I || cs);
    float t = 0.f;
    if (live) {
#pragma unroll 8
        for (int s = warp; s < slices; s += 8) t += part[(size_t)s * O * (I + 1) + q];
    }
    red[warp][lane] = t;
    __syncthreads();
    if (warp || !live) return;
    for (int w = 1; w < 8; ++w) t += red[w][lane];
    if (i < I) out[(size_t)o * I + i] = t;
    else cs[o] = t;
}

// O and I are multiples of 4 and the rows 16-byte aligned (channels and q/k
// columns of the models).
void launch_atb(int N, int O, int I, const float *G, const float *X, float *out, float *cs, float *part,
                cudaStream_t st) {
    if (O == 0 || I == 0) return;
    const int slices = std::max(1, std::min(ATB_SLICES, (N + 255) / 256));
    dim3 grid((O + ATB_T - 1) / ATB_T, (I + ATB_T - 1) / ATB_T, slices);
    k_atb_part<<<grid, 256, 0, st>>>(N, O, I, G, X, part, cs != nullptr, slices);
    count_launch();
    const int tot = O * (I + 1);
    k_atb_reduce<<<(tot + 31) / 32, 256, 0, st>>>(O, I, part, out, cs, slices);
    count_launch();
}

// ------------------------------------------- NC layer weight gradients
// With the layer factored over species (first.cu), A_i[lm][c] =
// nu sum_z emb[z][c] sum_k W_lkc T_i[z][lm][k], the gradients are
//   dW_lkc = nu sum_i sum_z emb[z][c] sum_m gA_i[lm][c] T_i[z][lm][k],
//   dU[t][c] = sum_i sum_m gV_i[t][m] A_i[1 + m][c],
//   gA_i = 2 A_i gq_i (+ for l = 1 sum_t U[t] gV_i[t][m]):
// no neighbour is visited again. Warps take atoms in a grid stride, lanes own
// C / 32 channels; each block adds its warps' sums in warp order into its row
// of `part`, and k_sum_rows adds the rows in a fixed order: deterministic.
// (49,152 atoms, C = 64: 68 + 14 us;
// 597 + 372 + 72 us when every edge was visited again and dU was
// summed by 64 blocks of its own.)
constexpr int WG_WARPS = 4;

template <int C>
__global__ void __launch_bounds__(WG_WARPS * 32) k_nc_layer_wgrad(NCLayerGradArgs g, float *__restrict__ part) {
    constexpr int K = 8, CPW = C / 32, NW = 2 * K * C, MAXL = 4;
    extern __shared__ float wg_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, S = g.n_species, Q = NW + g.n_l * C;
    float *red = wg_smem + warp * Q, *sE = wg_smem + WG_WARPS * Q, *sT = sE + S * C + warp * S * 32;
    for (int q = threadIdx.x; q < S * C; q += blockDim.x) sE[q] = __ldg(g.emb + q);
    __syncthreads();
    float wacc[2][K][CPW], uacc[MAXL][CPW];
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int u = 0; u < CPW; ++u) wacc[l][k][u] = 0.f;
#pragma unroll
    for (int h = 0; h < MAXL; ++h)
#pragma unroll
        for (int u = 0; u < CPW; ++u) uacc[h][u] = 0.f;
    const int c0 = lane * CPW;
    const int n = *g.err ? 0 : g.n_atoms;
    for (int i = blockIdx.x * WG_WARPS + warp; i < n; i += gridDim.x * WG_WARPS) {
        unsigned present = 0;
        for (int s = 0; s < S; ++s) {
            const float t = __ldg(g.T + ((size_t)i * S + s) * 32 + lane);   // [lm][k]
            sT[s * 32 + lane] = t;
            if (__any_sync(DMTS_FULL, t != 0.f)) present |= 1u << s;
        }
        float gA[4][CPW];
#pragma unroll
        for (int u = 0; u < CPW; ++u) {
            const int c = c0 + u;
            const float g0 = __ldg(g.gq + (size_t)i * 2 * C + c), g1 = __ldg(g.gq + (size_t)i * 2 * C + C + c);
            gA[0][u] = 2.f * __ldg(g.A + ((size_t)i * 4) * C + c) * g0;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const float A = __ldg(g.A + ((size_t)i * 4 + 1 + m) * C + c);
                float t = 2.f * A * g1;
#pragma unroll
                for (int h = 0; h < MAXL; ++h)
                    if (h < g.n_l) {
                        const float v = __ldg(g.gV + ((size_t)i * g.n_l + h) * 3 + m);
                        t = fmaf(__ldg(g.U + h * C + c), v, t);
                        uacc[h][u] = fmaf(v, A, uacc[h][u]);
                    }
                gA[1 + m][u] = t;
            }
        }
        __syncwarp();
        for (unsigned ms = present; ms; ms &= ms - 1) {
            const int s = __ffs(ms) - 1;
            const float *t = sT + s * 32;
            float e[CPW];
#pragma unroll
            for (int u = 0; u < CPW; ++u) e[u] = sE[s * C + c0 + u];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float t0 = t[k], t1 = t[K + k], t2 = t[2 * K + k], t3 = t[3 * K + k];
#pragma unroll
                for (int u = 0; u < CPW; ++u) {
                    wacc[0][k][u] = fmaf(e[u], gA[0][u] * t0, wacc[0][k][u]);
                    wacc[1][k][u] = fmaf(e[u], fmaf(gA[1][u], t1, fmaf(gA[2][u], t2, gA[3][u] * t3)), wacc[1][k][u]);
                }
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < CPW; ++u) {
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int k = 0; k < K; ++k) red[(l * K + k) * C + c0 + u] = g.nu * wacc[l][k][u];
#pragma unroll
        for (int h = 0; h < MAXL; ++h)
            if (h < g.n_l) red[NW + h * C + c0 + u] = uacc[h][u];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < Q; q += blockDim.x) {
        float t = wg_smem[q];
        for (int w = 1; w < WG_WARPS; ++w) t += wg_smem[w * Q + q];
        part[(size_t)blockIdx.x * Q + q] = t;
    }
}

// out[q] = sum over rows of part[row][q]: eight warps add every eighth row, in
// row order, and the eight sums are added in warp order. The first Qa sums go
// to `out`, the others to `out2`.
__global__ void __launch_bounds__(256) k_sum_rows(int Q, int rows, const float *__restrict__ part,
                                                  float *__restrict__ out, int Qa, float *__restrict__ out2) {
    __shared__ float red[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * 32 + lane;
    float t = 0.f;
    if (q < Q) {
#pragma unroll 4
        for (int r = warp; r < rows; r += 8) t += part[(size_t)r * Q + q];
    }
    red[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && q < Q) {
        for (int w = 1; w < 8; ++w) t += red[w][lane];
        if (q < Qa) out[q] = t;
        else out2[q - Qa] = t;
    }
}

void launch_nc_layer_wgrad(int C, const NCLayerGradArgs &a, float *part, float *dW, float *dU, cudaStream_t st) {
    if (a.n_atoms == 0) return;
    const int blocks = std::max(1, std::min(WG_BLOCKS, (a.n_atoms + WG_WARPS - 1) / WG_WARPS));
    const int NW = 2 * 8 * C, Q = NW + a.n_l * C;
    const size_t smem = sizeof(float) * (WG_WARPS * (Q + (size_t)a.n_species * 32) + (size_t)a.n_species * C);
    if (C == 32) k_nc_layer_wgrad<32><<<blocks, WG_WARPS * 32, smem, st>>>(a, part);
    else if (C == 64) k_nc_layer_wgrad<64><<<blocks, WG_WARPS * 32, smem, st>>>(a, part);
    else return;
    count_launch();
    k_sum_rows<<<(Q + 31) / 32, 256, 0, st>>>(Q, blocks, part, dW, NW, dU);
    count_launch();
}

__global__ void k_distill_residual(int n, const float *F, const float *T, float *g, float *sq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float d = F[3 * i + q] - T[3 * i + q];
        g[3 * i + q] = 2.f * d;
        s = fmaf(d, d, s);
    }
    sq[i] = s;
}

void launch_distill_residual(int n, const float *F, const float *T, float *g, float *sq, cudaStream_t st) {
    if (n == 0) return;
    k_distill_residual<<<(n + 255) / 256, 256, 0, st>>>(n, F, T, g, sq);
    count_launch();
}

// Adam (Kingma & Ba), beta1 0.9, beta2 0.999, eps 1e-8, bias-corrected.
__global__ void k_adam(int n, float *w, const float *grad, float *m, float *v, float lr, float c1, float c2,
                       __nv_bfloat16 *w_bf, int kd) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gr = grad[i];
    const float mi = 0.9f * m[i] + 0.1f * gr, vi = 0.999f * v[i] + 0.001f * gr * gr;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    w[i] = wi;
    if (w_bf) st_split(w_bf, (size_t)(i / kd), kd, i % kd, wi);
}

void launch_adam(int n, float *w, const float *grad, float *m, float *v, float lr, int step, __nv_bfloat16 *w_bf,
                 int kd, cudaStream_t st) {
    if (n == 0) return;
    const float c1 = 1.f - powf(0.9f, (float)step), c2 = 1.f - powf(0.999f, (float)step);
    k_adam<<<(n + 255) / 256, 256, 0, st>>>(n, w, grad, m, v, lr, c1, c2, w_bf, kd);
    count_launch();
}

}  // namespace dmts
