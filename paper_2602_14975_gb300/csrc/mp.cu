// Message-passing layers after the first (first.cu): edge embedding (Bessel x envelope, real SH),
// segmented scatter-sum with one warp per receiver, and the adjoint (forces
// and feature gradients): each pair's force once, from its lower atom, in
// fixed point; each atom's sender-role gradient gathered over its row of the
// symmetric neighbour list. Node-level MLP contractions: SIMT fp32 GEMM with
// fused epilogues.
#include <algorithm>

#include "epilogue.cuh"
#include "mp.cuh"
#include "pack.cuh"
#include "ptx.cuh"

namespace dmts {

constexpr int MP_WARPS = 4;

// ------------------------------------------------------------------ forward
// Warp per receiver i, lane owns CPW consecutive channels c = lane*CPW + u.
// Active edges (r < rc) of the row are compacted 32 at a time into shared
// memory with their embedding (f_c B_k, Y_lm); every lane then sweeps them.
// C channels are split over SPLIT thread blocks (blockIdx.y = part): a warp
// owns CW = C / SPLIT channels, offset co = part * CW.
template <int C, int LMAX, int K, int SPLIT>
__global__ void __launch_bounds__(MP_WARPS * 32) k_mp_fwd(EdgeGeom g, LayerIO io) {
    constexpr int NL = LMAX + 1, NLM = NL * NL, CW = C / SPLIT, CPW = CW / 32;
    using T = typename Pack<CPW>::T;
    constexpr int NP = Pack<CPW>::NP, PW = Pack<CPW>::W;
    constexpr int RS = (K + NLM) | 1;   // odd record stride: conflict-free writes
    constexpr int FWD_UNROLL = LMAX >= 2 ? 2 : 4;   // edges in flight per lane (registers allowing)
    const int co = blockIdx.y * CW;
    __shared__ T sh_r[MP_WARPS][32][RS];
    __shared__ int sh_j[MP_WARPS][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wi = blockIdx.x * MP_WARPS + warp;
    if (wi >= g.n_atoms || *io.err) return;
    const int i = g.order ? __ldg(g.order + wi) : wi;   // spatially sorted: neighbours shared in cache

    T W[NL][K][NP];
#pragma unroll
    for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int k = 0; k < K; ++k) ldp<CPW>(io.wrad + (l * K + k) * C + co + lane * CPW, W[l][k]);
    T acc[NLM][NP];
#pragma unroll
    for (int lm = 0; lm < NLM; ++lm)
#pragma unroll
        for (int p = 0; p < NP; ++p) acc[lm][p] = vdup<T>(0.f);

    const int rep = g.atom_rep[i];
    const float bx = g.box[3 * rep], by = g.box[3 * rep + 1], bz = g.box[3 * rep + 2];
    const float ibx = bx > 0.f ? 1.f / bx : 0.f, iby = by > 0.f ? 1.f / by : 0.f, ibz = bz > 0.f ? 1.f / bz : 0.f;
    const float xi = g.x[3 * i], yi = g.x[3 * i + 1], zi = g.x[3 * i + 2];
    const float rc2 = g.rc * g.rc;
    const int beg = g.row_ptr[i], end = g.row_ptr[i + 1];
    for (int base = beg; base < end; base += 32) {
        const int e = base + lane;
        bool act = false;
        int j = 0;
        float dx = 0.f, dy = 0.f, dz = 0.f, r2 = 0.f;
        if (e < end) {
            j = __ldg(g.col + e);
            dx = min_img(__ldg(g.x + 3 * j) - xi, bx, ibx);
            dy = min_img(__ldg(g.x + 3 * j + 1) - yi, by, iby);
            dz = min_img(__ldg(g.x + 3 * j + 2) - zi, bz, ibz);
            r2 = dx * dx + dy * dy + dz * dz;
            act = r2 < rc2;
        }
        const unsigned m = __ballot_sync(DMTS_FULL, act);
        if (act) {
            const int pos = __popc(m & ((1u << lane) - 1u));
            T *rec = sh_r[warp][pos];
            const float r = sqrtf(r2), inv = 1.f / r;
            float du;
            const float fc = envelope(r * g.inv_rc, g.p, &du);
            float B[K];
            bessel<K, false>(r, g.inv_rc, g.bnorm, B, nullptr);
#pragma unroll
            for (int k = 0; k < K; ++k) rec[k] = vdup<T>(fc * B[k]);
            float Y[NLM];
            sph<LMAX>(dx * inv, dy * inv, dz * inv, Y);
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) rec[K + lm] = vdup<T>(Y[lm]);
            sh_j[warp][pos] = j;
        }
        __syncwarp();
        const int na = __popc(m);
#pragma unroll FWD_UNROLL
        for (int t = 0; t < na; ++t) {
            const int jt = sh_j[warp][t];
            const T *rec = sh_r[warp][t];
            T sj[NP];
            ldp<CPW>(io.s + (size_t)jt * C + co + lane * CPW, sj);
            T b[K], y[NLM];
#pragma unroll
            for (int k = 0; k < K; ++k) b[k] = rec[k];
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) y[lm] = rec[K + lm];
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    T Ra = vdup<T>(0.f), Rb = vdup<T>(0.f);
#pragma unroll
                    for (int k = 0; k < K; k += 2) {
                        Ra = vfma(W[l][k][p], b[k], Ra);
                        Rb = vfma(W[l][k + 1][p], b[k + 1], Rb);
                    }
                    const T R = vadd(Ra, Rb);
                    const T msg = vmul(R, sj[p]);
#pragma unroll
                    for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) acc[lm][p] = vfma(msg, y[lm], acc[lm][p]);
                }
        }
        __syncwarp();
    }
    const T nu = vdup<T>(io.nu);
    T qv[NL][NP];
#pragma unroll
    for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int p = 0; p < NP; ++p) qv[l][p] = vdup<T>(0.f);
#pragma unroll
    for (int lm = 0; lm < NLM; ++lm) {
        const int l = lm == 0 ? 0 : (lm < 4 ? 1 : 2);
        T a[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            a[p] = vmul(nu, acc[lm][p]);
            qv[l][p] = vfma(a[p], a[p], qv[l][p]);
        }
        stp<CPW>(io.A + ((size_t)i * NLM + lm) * C + co + lane * CPW, a);
    }
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        stp<CPW>(io.q + (size_t)i * NL * C + l * C + co + lane * CPW, qv[l]);
        if (io.q_bf16) {
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int hh = 0; hh < PW; ++hh)
                    st_split(io.q_bf16, i, NL * C, l * C + co + lane * CPW + p * PW + hh, vget(qv[l][p], hh));
        }
    }
}

// ----------------------------------------------------------------- adjoint
// For atom a and a neighbour j (n = n_aj, r = r_aj), with
//   Gam[c][lm] = gA_a[lm][c] s_j[c] + (-1)^l gA_j[lm][c] s_a[c],
// the pair's force on a (both edges a <- j and j <- a) is
//   f_aj = nu ( rho n + sum_lm beta_lm dY_lm/dd ),
//   rho = sum_c sum_l R'_lc sum_m Gam Y_lm,  beta_lm = sum_c Gam R_lc,
// and the feature gradient of the sender role is
//   g_s_a[c] += nu sum_j sum_l (-1)^l R_lc sum_m gA_j[lm][c] Y_lm.
// Edge j -> a has d_ja = -d_aj and Y_lm(-n) = (-1)^l Y_lm(n), so
// Gam_ja = (-1)^l Gam_aj and dY_lm/dd at -d is -(-1)^l dY_lm/dd at d: the
// pair terms are antisymmetric, f_ja = -f_aj. Each pair's force is formed
// once, by the warp of its lower atom a < j, and enters F_a with + and F_j
// with -, in 32.32 fixed point (exact, order-independent sums; every pair's
// two terms cancel exactly), and so does its virial term. A lower
// neighbour j < a contributes only its sender-role term to g_s_a (R, no R',
// no force).
//
// Shared memory per block (one warp; 21.4 KB at C = 128, l_max = 2): 32 edge
// records of packs (f_c B_k, its r-derivative, Y_lm) and of scalars
// (dY_lm/dd, n, and r for the virial), the receiver's gA_a as packs, the 32
// neighbour indices, and the lanes' shares of the force of FT pairs
// (transposed so that one lane adds up each pair).
constexpr int FT = 16;   // pairs per force reduction
// One warp per block: how many upper neighbours an atom has varies from atom
// to atom, and a block keeps its registers and shared memory until its
// slowest warp is done, so single-warp blocks keep the SM's eight warp slots
// busy (255 registers a thread allow eight warps per SM either way).
constexpr int BWD_WARPS = 1;

template <int C, int LMAX, int K, bool VIR>
struct BwdSmem {
    static constexpr int NL = LMAX + 1, NLM = NL * NL, CPW = C / 32;
    using T = typename Pack<CPW>::T;
    static constexpr int NP = Pack<CPW>::NP;
    static constexpr int RS = (2 * K + NLM) | 1;
    static constexpr int GS = (3 * NLM + 3 + (VIR ? 1 : 0)) | 1;
    static constexpr size_t r_bytes = sizeof(T) * BWD_WARPS * 32 * RS;
    static constexpr size_t ga_bytes = sizeof(T) * BWD_WARPS * NLM * NP * 32;
    static constexpr size_t g_bytes = sizeof(float) * BWD_WARPS * 32 * GS;
    static constexpr size_t j_bytes = sizeof(int) * BWD_WARPS * 32;
    static constexpr size_t f_bytes = sizeof(float) * BWD_WARPS * 3 * FT * 33;
    static constexpr size_t bytes = r_bytes + ga_bytes + g_bytes + j_bytes + f_bytes;
};

template <int C, int LMAX, int K, bool VIR>
__global__ void __launch_bounds__(BWD_WARPS * 32) k_mp_bwd(EdgeGeom g, LayerIO io) {
    using S = BwdSmem<C, LMAX, K, VIR>;
    using T = typename S::T;
    constexpr int NL = S::NL, NLM = S::NLM, CPW = S::CPW, NP = S::NP, PW = Pack<CPW>::W;
    constexpr int RS = S::RS, GS = S::GS;
    extern __shared__ __align__(16) unsigned char mp_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T (*sh_r)[RS] = reinterpret_cast<T (*)[RS]>(mp_smem) + warp * 32;
    T (*sh_ga)[NP * 32] = reinterpret_cast<T (*)[NP * 32]>(mp_smem + S::r_bytes) + warp * NLM;
    float (*sh_g)[GS] = reinterpret_cast<float (*)[GS]>(mp_smem + S::r_bytes + S::ga_bytes) + warp * 32;
    int *sh_j = reinterpret_cast<int *>(mp_smem + S::r_bytes + S::ga_bytes + S::g_bytes) + warp * 32;
    float (*sh_f)[FT][33] =
        reinterpret_cast<float (*)[FT][33]>(mp_smem + S::r_bytes + S::ga_bytes + S::g_bytes + S::j_bytes) + warp * 3;
    const int wa = blockIdx.x * BWD_WARPS + warp;
    if (wa >= g.n_atoms || *io.err) return;
    const int a = g.order ? __ldg(g.order + wa) : wa;

    T W[NL][K][NP];
#pragma unroll
    for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int k = 0; k < K; ++k) ldp<CPW>(io.wrad + (l * K + k) * C + lane * CPW, W[l][k]);
#pragma unroll
    for (int lm = 0; lm < NLM; ++lm) {
        T t[NP];
        ldp<CPW>(io.gA + ((size_t)a * NLM + lm) * C + lane * CPW, t);
#pragma unroll
        for (int p = 0; p < NP; ++p) sh_ga[lm][p * 32 + lane] = t[p];
    }
    T sa[NP], san[NP], gse[NP], gso[NP];   // s_a, -s_a; sender-role sums over even and odd l
    ldp<CPW>(io.s + (size_t)a * C + lane * CPW, sa);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        san[p] = vneg(sa[p]);
        gse[p] = vdup<T>(0.f);
        gso[p] = vdup<T>(0.f);
    }
    // a's side of its pairs, fixed point (on the lanes that add up a pair)
    long long oa[3] = {0, 0, 0}, ow = 0;
    bool bad = false;   // a pair term outside the fixed-point range (or not finite)

    const int rep = g.atom_rep[a];
    const float bx = g.box[3 * rep], by = g.box[3 * rep + 1], bz = g.box[3 * rep + 2];
    const float ibx = bx > 0.f ? 1.f / bx : 0.f, iby = by > 0.f ? 1.f / by : 0.f, ibz = bz > 0.f ? 1.f / bz : 0.f;
    const float xa = g.x[3 * a], ya = g.x[3 * a + 1], za = g.x[3 * a + 2];
    const float rc2 = g.rc * g.rc;
    const int beg = g.row_ptr[a], end = g.row_ptr[a + 1];
    __syncwarp();
    for (int base = beg; base < end; base += 32) {
        const int e = base + lane;
        bool act = false;
        int j = 0;
        float dx = 0.f, dy = 0.f, dz = 0.f, r2 = 0.f;
        if (e < end) {
            j = __ldg(g.col + e);
            dx = min_img(__ldg(g.x + 3 * j) - xa, bx, ibx);
            dy = min_img(__ldg(g.x + 3 * j + 1) - ya, by, iby);
            dz = min_img(__ldg(g.x + 3 * j + 2) - za, bz, ibz);
            r2 = dx * dx + dy * dy + dz * dz;
            act = r2 < rc2;
        }
        // lower neighbours (j < a) first, then the upper ones (the pairs this
        // warp owns): rows are ascending, so g_s_a takes its terms in row
        // order whatever the chunk boundaries (which move with the list's
        // skin entries)
        const bool up = act && j > a, lo = act && j < a;
        const unsigned mu = __ballot_sync(DMTS_FULL, up), ml = __ballot_sync(DMTS_FULL, lo);
        const int n_up = __popc(mu), n_lo = __popc(ml);
        if (up || lo) {
            const unsigned lt = (1u << lane) - 1u;
            const int pos = lo ? __popc(ml & lt) : n_lo + __popc(mu & lt);
            T *rec = sh_r[pos];
            float *ge = sh_g[pos];
            const float r = sqrtf(r2), inv = 1.f / r;
            float du;
            const float fc = envelope(r * g.inv_rc, g.p, &du);
            const float dfc = du * g.inv_rc;
            float B[K], dB[K];
            bessel<K, true>(r, g.inv_rc, g.bnorm, B, dB);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                rec[k] = vdup<T>(fc * B[k]);
                rec[K + k] = vdup<T>(dfc * B[k] + fc * dB[k]);
            }
            const float nx = dx * inv, ny = dy * inv, nz = dz * inv;
            float Y[NLM], dY[3 * NLM];
            sph<LMAX>(nx, ny, nz, Y);
            sph_grad<LMAX>(nx, ny, nz, inv, dY);
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) rec[2 * K + lm] = vdup<T>(Y[lm]);
#pragma unroll
            for (int q = 0; q < 3 * NLM; ++q) ge[q] = dY[q];
            ge[3 * NLM] = nx;
            ge[3 * NLM + 1] = ny;
            ge[3 * NLM + 2] = nz;
            if (VIR) ge[3 * NLM + 3] = r;
            sh_j[pos] = j;
        }
        __syncwarp();
        // lower neighbours: the sender-role gradient only
#pragma unroll 2
        for (int t = 0; t < n_lo; ++t) {
            const int jt = sh_j[t];
            const T *rec = sh_r[t];
            T gj[NLM][NP];
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) ldp<CPW>(io.gA + ((size_t)jt * NLM + lm) * C + lane * CPW, gj[lm]);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    T s0 = vdup<T>(0.f), s2 = vdup<T>(0.f);
#pragma unroll
                    for (int k = 0; k < K; k += 2) {
                        s0 = vfma(W[l][k][p], rec[k], s0);
                        s2 = vfma(W[l][k + 1][p], rec[k + 1], s2);
                    }
                    const T R = vadd(s0, s2);
                    T wl = vdup<T>(0.f);
#pragma unroll
                    for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) wl = vfma(gj[lm][p], rec[2 * K + lm], wl);
                    if (l & 1) gso[p] = vfma(R, wl, gso[p]);
                    else gse[p] = vfma(R, wl, gse[p]);
                }
            }
        }
        for (int t0 = n_lo; t0 < n_lo + n_up; t0 += FT) {
            const int t1 = min(n_lo + n_up, t0 + FT);
#pragma unroll 2
            for (int t = t0; t < t1; ++t) {
                const int jt = sh_j[t];
                const T *rec = sh_r[t];
                const float *ge = sh_g[t];
                T sj[NP];
                ldp<CPW>(io.s + (size_t)jt * C + lane * CPW, sj);
                T gj[NLM][NP];
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) ldp<CPW>(io.gA + ((size_t)jt * NLM + lm) * C + lane * CPW, gj[lm]);
                T y[NLM];
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) y[lm] = rec[2 * K + lm];
                T rho = vdup<T>(0.f), beta[NLM];
#pragma unroll
                for (int lm = 0; lm < NLM; ++lm) beta[lm] = vdup<T>(0.f);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    T R[NL], Rp[NL];
#pragma unroll
                    for (int l = 0; l < NL; ++l) {
                        T s0 = vdup<T>(0.f), s1 = vdup<T>(0.f), s2 = vdup<T>(0.f), s3 = vdup<T>(0.f);
#pragma unroll
                        for (int k = 0; k < K; k += 2) {
                            s0 = vfma(W[l][k][p], rec[k], s0);
                            s1 = vfma(W[l][k][p], rec[K + k], s1);
                            s2 = vfma(W[l][k + 1][p], rec[k + 1], s2);
                            s3 = vfma(W[l][k + 1][p], rec[K + k + 1], s3);
                        }
                        R[l] = vadd(s0, s2);
                        Rp[l] = vadd(s1, s3);
                    }
#pragma unroll
                    for (int l = 0; l < NL; ++l) {
                        const T sas = (l & 1) ? san[p] : sa[p];
                        T tl = vdup<T>(0.f), wl = vdup<T>(0.f);
#pragma unroll
                        for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                            const T gam = vfma(sh_ga[lm][p * 32 + lane], sj[p], vmul(gj[lm][p], sas));
                            tl = vfma(gam, y[lm], tl);
                            beta[lm] = vfma(gam, R[l], beta[lm]);
                            wl = vfma(gj[lm][p], y[lm], wl);
                        }
                        rho = vfma(Rp[l], tl, rho);
                        if (l & 1) gso[p] = vfma(R[l], wl, gso[p]);
                        else gse[p] = vfma(R[l], wl, gse[p]);
                    }
                }
                // this lane's share (its channels) of the pair's force on a
                const float rh = vsum(rho);
                float ex = rh * ge[3 * NLM], ey = rh * ge[3 * NLM + 1], ez = rh * ge[3 * NLM + 2];
#pragma unroll
                for (int lm = 1; lm < NLM; ++lm) {
                    const float bl = vsum(beta[lm]);
                    ex = fmaf(bl, ge[3 * lm], ex);
                    ey = fmaf(bl, ge[3 * lm + 1], ey);
                    ez = fmaf(bl, ge[3 * lm + 2], ez);
                }
                sh_f[0][t - t0][lane] = ex;
                sh_f[1][t - t0][lane] = ey;
                sh_f[2][t - t0][lane] = ez;
            }
            __syncwarp();
            // pair t0 + u: lanes u and u + 16 add up lanes 0-15 and 16-31 of
            // its shares (conflict-free: row stride 33), then lane u the two
            // halves, in a fixed order
            const int u = lane & (FT - 1), h = lane / FT;
            const bool own = t0 + u < t1;
            float px = 0.f, py = 0.f, pz = 0.f;
            if (own) {
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    px += sh_f[0][u][16 * h + q];
                    py += sh_f[1][u][16 * h + q];
                    pz += sh_f[2][u][16 * h + q];
                }
            }
            px += __shfl_down_sync(DMTS_FULL, px, 16);
            py += __shfl_down_sync(DMTS_FULL, py, 16);
            pz += __shfl_down_sync(DMTS_FULL, pz, 16);
            if (own && h == 0) {
                const int jt = sh_j[t0 + u];
                px *= io.nu;
                py *= io.nu;
                pz *= io.nu;
                if (fix_ok(px) && fix_ok(py) && fix_ok(pz)) {
                    const long long qx = to_fix(px), qy = to_fix(py), qz = to_fix(pz);
                    oa[0] += qx;
                    oa[1] += qy;
                    oa[2] += qz;
                    unsigned long long *fj = io.Ffix + 3 * (size_t)jt;
                    fix_add(fj, -qx);
                    fix_add(fj + 1, -qy);
                    fix_add(fj + 2, -qz);
                    if (VIR) {
                        // virial proxy: dU/dd . d of the pair, half to each end
                        const float *ge = sh_g[t0 + u];
                        const float wp = 0.5f * ge[3 * NLM + 3] * (px * ge[3 * NLM] + py * ge[3 * NLM + 1] + pz * ge[3 * NLM + 2]);
                        if (fix_ok(wp)) {
                            const long long qw = to_fix(wp);
                            ow += qw;
                            fix_add(io.Wfix + jt, qw);
                        } else {
                            bad = true;
                        }
                    }
                } else {
                    bad = true;
                }
            }
            __syncwarp();
        }
        __syncwarp();
    }
    // a's side: the integer sums of the lanes that added up its pairs
    oa[0] = warp_sum_fix(oa[0]);
    oa[1] = warp_sum_fix(oa[1]);
    oa[2] = warp_sum_fix(oa[2]);
    if (VIR) ow = warp_sum_fix(ow);
    if (__any_sync(DMTS_FULL, bad) && lane == 0) set_error(io.err, (int)DMTS_E_NONFINITE);
    if (lane == 0) {
        unsigned long long *fa = io.Ffix + 3 * (size_t)a;
        fix_add(fa, oa[0]);
        fix_add(fa + 1, oa[1]);
        fix_add(fa + 2, oa[2]);
        if (VIR) fix_add(io.Wfix + a, ow);
    }
    T gin[NP], gout[NP];
    ldp<CPW>(io.gs_in + (size_t)a * C + lane * CPW, gin);
#pragma unroll
    for (int p = 0; p < NP; ++p) gout[p] = vfma(vdup<T>(io.nu), vsub(gse[p], gso[p]), gin[p]);
    stp<CPW>(io.gs_out + (size_t)a * C + lane * CPW, gout);
    if (io.gs_out_bf16) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int hh = 0; hh < PW; ++hh)
                st_split(io.gs_out_bf16, a, C, lane * CPW + p * PW + hh, vget(gout[p], hh));
    }
}

// One thread per atom: the adjoint's fixed-point forces (and virial) -> fp32,
// the words cleared for the next evaluation (also after an aborted one).
__global__ void k_fix_convert(int n, unsigned long long *__restrict__ Ffix, float *__restrict__ F,
                              unsigned long long *__restrict__ Wfix, float *__restrict__ W) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long q = (long long)Ffix[3 * (size_t)i + c];
        Ffix[3 * (size_t)i + c] = 0ull;
        F[3 * (size_t)i + c] = fix_to_float(q);
    }
    if (Wfix) {
        const long long q = (long long)Wfix[i];
        Wfix[i] = 0ull;
        W[i] = fix_to_float(q);
    }
}

void launch_fix_convert(int n, unsigned long long *Ffix, float *F, unsigned long long *Wfix, float *W,
                        cudaStream_t st) {
    if (n == 0) return;
    k_fix_convert<<<(n + 255) / 256, 256, 0, st>>>(n, Ffix, F, Wfix, W);
    count_launch();
}

// In the forward pass 128 channels are split over two blocks (64 per warp):
// half the registers, twice the warps in flight to hide the neighbour loads.
template <int C, int LMAX>
static void fwd_c(const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    constexpr int SP = C >= 128 ? 2 : 1;
    const int blocks = (g.n_atoms + MP_WARPS - 1) / MP_WARPS;
    k_mp_fwd<C, LMAX, 8, SP><<<dim3(blocks, SP), MP_WARPS * 32, 0, st>>>(g, io);
    count_launch();
}

template <int C, int LMAX, bool VIR>
static void bwd_launch(const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    constexpr size_t smem = BwdSmem<C, LMAX, 8, VIR>::bytes;
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_mp_bwd<C, LMAX, 8, VIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int blocks = (g.n_atoms + BWD_WARPS - 1) / BWD_WARPS;
    k_mp_bwd<C, LMAX, 8, VIR><<<blocks, BWD_WARPS * 32, smem, st>>>(g, io);
    count_launch();
}

// The virial variant (io.Wfix set) is a separate instantiation, so that the
// other carries no register or instruction it does not use.
template <int C, int LMAX>
static void bwd_c(const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    io.Wfix ? bwd_launch<C, LMAX, true>(g, io, st) : bwd_launch<C, LMAX, false>(g, io, st);
}

void launch_mp_fwd(int C, int lmax, int K, const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    (void)K;
    if (g.n_atoms == 0) return;
    DMTS_DISPATCH(fwd_c, C, lmax, g, io, st);
}

void launch_mp_bwd(int C, int lmax, int K, const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    (void)K;
    if (g.n_atoms == 0) return;
    DMTS_DISPATCH(bwd_c, C, lmax, g, io, st);
}

// -------------------------------------------------------------------- GEMM
// fp32 SIMT contraction. A CTA computes a BM x BN tile; K is walked in chunks
// of 32, GEMM_STAGES of them in flight (16-byte asynchronous copies, zero
// filled past M, N and K). Both tiles are kept k-contiguous (row stride 36:
// the eight rows a quarter-warp reads with 16-byte loads lie in distinct
// banks), so that a packed operand is two consecutive k of one row: every
// output sums its even and its odd k in one packed accumulator and adds the
// two at the end, with no register moves. The order does not depend on the
// tile, so an atom's result does not depend on the batch it is in.
// At 23,558 rows (N = K = 128) a contraction takes 27 us, 29 TFLOP/s (the
// one-chunk 64 x 64 kernel it replaced: 14 contractions of a conservative call
// 1336 -> 777 us); bound by shared-memory wavefronts and the epilogue's global
// accesses. At 192 rows it is bound by latency: 17 -> 7.5 us per call.
constexpr int GEMM_KC = 32, GEMM_LD = GEMM_KC + 4, GEMM_STAGES = 3;

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) k_gemm_f32(int M, int N, int K, const float *__restrict__ Act,
                                                                   const float *__restrict__ W, int trans, int vec, Epi e) {
    constexpr int THREADS = (BM / TM) * (BN / TN), TY = BM / TM, TX = BN / TN, CH = GEMM_KC / 4;
    extern __shared__ __align__(16) float gemm_smem[];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int nk = (K + GEMM_KC - 1) / GEMM_KC;
    auto As = [&](int s) { return gemm_smem + s * (BM + BN) * GEMM_LD; };
    auto Bs = [&](int s) { return gemm_smem + (s * (BM + BN) + BM) * GEMM_LD; };
    auto load = [&](int c) {
        float *a = As(c % GEMM_STAGES), *b = Bs(c % GEMM_STAGES);
        const int k0 = c * GEMM_KC;
        for (int q = tid; q < BM * CH; q += THREADS) {
            const int r = q / CH, k = k0 + 4 * (q % CH);
            const bool ok = m0 + r < M && k < K;
            cp_async16(smem_u32(a + r * GEMM_LD + 4 * (q % CH)), ok ? Act + (size_t)(m0 + r) * K + k : Act, ok);
        }
        if (trans) {
            for (int q = tid; q < BN * CH; q += THREADS) {
                const int r = q / CH, k = k0 + 4 * (q % CH);
                const bool ok = n0 + r < N && k < K;
                cp_async16(smem_u32(b + r * GEMM_LD + 4 * (q % CH)), ok ? W + (size_t)(n0 + r) * K + k : W, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // W [K][N] (trans = 0): rows along n, through registers and transposed
    // into shared memory; loaded before a chunk's arithmetic, stored after it
    constexpr int WPT = GEMM_KC * BN / THREADS;
    float wr[WPT];
    auto load_w = [&](int c) {
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
            const int q = tid + u * THREADS, r = q % BN, k = c * GEMM_KC + q / BN;
            wr[u] = (n0 + r < N && k < K) ? __ldg(W + (size_t)k * N + n0 + r) : 0.f;
        }
    };
    auto store_w = [&](int c) {
        float *b = Bs(c % GEMM_STAGES);
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
            const int q = tid + u * THREADS;
            b[q % BN * GEMM_LD + q / BN] = wr[u];
        }
    };
    float2 acc[TM][TN];
#pragma unroll
    for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < TN; ++q) acc[p][q] = make_float2(0.f, 0.f);
    for (int c = 0; c < GEMM_STAGES - 1; ++c) {
        if (c < nk) {
            load(c);
            if (!trans) {
                load_w(c);
                store_w(c);
            }
        } else {
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    }
    for (int c = 0; c < nk; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(GEMM_STAGES - 2) : "memory");
        __syncthreads();   // chunk c landed for every thread; the buffer of chunk c - 1 is free
        const bool more = c + GEMM_STAGES - 1 < nk;
        if (more) {
            load(c + GEMM_STAGES - 1);
            if (!trans) load_w(c + GEMM_STAGES - 1);
        } else {
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        const float *a = As(c % GEMM_STAGES) + ty * GEMM_LD, *b = Bs(c % GEMM_STAGES) + tx * GEMM_LD;
#pragma unroll
        for (int k = 0; k < GEMM_KC; k += 4) {
            float4 av[TM];
#pragma unroll
            for (int p = 0; p < TM; ++p) av[p] = *reinterpret_cast<const float4 *>(a + p * TY * GEMM_LD + k);
#pragma unroll
            for (int q = 0; q < TN; ++q) {
                const float4 bv = *reinterpret_cast<const float4 *>(b + q * TX * GEMM_LD + k);
#pragma unroll
                for (int p = 0; p < TM; ++p) {
                    acc[p][q] = __ffma2_rn(make_float2(av[p].x, av[p].y), make_float2(bv.x, bv.y), acc[p][q]);
                    acc[p][q] = __ffma2_rn(make_float2(av[p].z, av[p].w), make_float2(bv.z, bv.w), acc[p][q]);
                }
            }
        }
        if (more && !trans) store_w(c + GEMM_STAGES - 1);
    }
    // the tile through shared memory, so that the epilogue's accesses are
    // whole rows whatever its mode
    cp_async_wait_all();
    __syncthreads();
    constexpr int LD = BN + 1;
    static_assert(BM * LD <= GEMM_STAGES * (BM + BN) * GEMM_LD, "the staged tile reuses the pipeline buffers");
#pragma unroll
    for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < TN; ++q) gemm_smem[(ty + p * TY) * LD + tx + q * TX] = acc[p][q].x + acc[p][q].y;
    __syncthreads();
    const int rows = min(BM, M - m0), cols = min(BN, N - n0);
    if (vec) epilogue_tile_v4(e, N, rows, m0, n0, cols, gemm_smem, LD);
    else epilogue_tile(e, N, rows, m0, n0, cols, gemm_smem, LD);
}

template <int BM, int BN, int TM, int TN>
static void gemm_f32_launch(int M, int N, int K, const float *Act, const float *W, int trans, const Epi &e,
                            cudaStream_t st) {
    constexpr size_t smem = sizeof(float) * GEMM_STAGES * (BM + BN) * GEMM_LD;
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_gemm_f32<BM, BN, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
    k_gemm_f32<BM, BN, TM, TN><<<grid, (BM / TM) * (BN / TN), smem, st>>>(M, N, K, Act, W, trans, N % 4 == 0 && epilogue_vectorizable(e), e);
    count_launch();
}

// K is a multiple of 4 and both operands are 16-byte aligned (every
// contraction of the models: rows of C, (l_max + 1) C or 2 H n_c floats).
void launch_gemm_f32(int M, int N, int K, const float *Act, const float *W, int trans, const Epi &e,
                     cudaStream_t st) {
    if (M == 0) return;
    static int n_sm = 0;
    if (!n_sm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        n_sm = std::max(n_sm, 1);
    }
    // small tiles until the large ones give every SM two CTAs: at 4,000 rows
    // (N = K = 128) 10.4 us against 8.3 (plain) and 12.3 against 12.4 (SiLU
    // epilogue), at 192 rows 6.2 against 8.3, at 23,558 rows 41 against 27
    if ((long long)((M + 63) / 64) * ((N + 63) / 64) >= 2LL * n_sm) gemm_f32_launch<64, 64, 4, 4>(M, N, K, Act, W, trans, e, st);
    else gemm_f32_launch<16, 32, 2, 2>(M, N, K, Act, W, trans, e, st);
}

// -------------------------------------------------- per-replica FP64 sums
__global__ void k_replica_sum(const float *__restrict__ v, const int *__restrict__ rep_off,
                              double *__restrict__ out, int accumulate) {
    __shared__ double red[32];
    const int r = blockIdx.x;
    const int beg = rep_off[r], end = rep_off[r + 1];
    double acc = 0.0;
    const int stride = blockDim.x;
    for (int i0 = beg + threadIdx.x; i0 < end; i0 += 8 * stride) {
        float t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = i0 + u * stride < end ? v[i0 + u * stride] : 0.f;
        float b = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) b += t[u];
        acc += (double)b;
    }
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        t = warp_sum_d(t);
        if (threadIdx.x == 0) out[r] = accumulate ? out[r] + t : t;
    }
}

void launch_replica_sum(const float *v, const int *rep_off, int n_rep, double *out, int accumulate,
                        cudaStream_t st) {
    if (n_rep == 0) return;
    k_replica_sum<<<n_rep, 1024, 0, st>>>(v, rep_off, out, accumulate);
    count_launch();
}

}  // namespace dmts
