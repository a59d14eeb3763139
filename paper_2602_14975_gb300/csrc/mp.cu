// Message-passing layers after the first (first.cu): edge embedding (Bessel x envelope, real SH),
// segmented scatter-sum with one warp per receiver, and the adjoint (forces
// and feature gradients): each pair's force once, from its lower atom, in
// fixed point; each atom's sender-role gradient gathered over its row of the
// symmetric neighbour list. Node-level MLP contractions: SIMT fp32 GEMM with
// fused epilogues.
#include <algorithm>

#include "edge.cuh"
#include "epilogue.cuh"
#include "launch.cuh"
#include "mp.cuh"
#include "pack.cuh"
#include "ptx.cuh"

namespace dmts {

constexpr int MP_WARPS = 4;
constexpr unsigned kOneWave = 1024;   // warps that are all resident from the start (launch.cuh)

// ------------------------------------------------------------------ forward
// Warp per receiver i, lane owns CPW consecutive channels c = lane*CPW + u.
// Active edges (r < rc) of the row are compacted 32 at a time into shared
// memory with their embedding (f_c B_k, Y_lm); every lane then sweeps them.
// C channels are split over SPLIT thread blocks (blockIdx.y = part): a warp
// owns CW = C / SPLIT channels, offset co = part * CW.
template <int C, int LMAX, int K, int SPLIT>
__global__ void __launch_bounds__(MP_WARPS * 32) k_mp_fwd(EdgeGeom g, LayerIO io) {
    dep_entry(gridDim.x <= kOneWave / MP_WARPS);
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
// One warp per block and atom: how many upper neighbours an atom has varies,
// and a block keeps its registers until its slowest warp is done. What bounds
// it: latency and issue at eight warps per SM (24 packs of radial weights live
// in registers), 288 packed FMA of two cycles per pair, and the L1 data path
// (the neighbours' rows gA_j, s_j, edge records). So the records are read 16
// bytes at a time, the direction derivative is formed from n instead of nine
// stored gradients, and the next chunk's candidates are loaded a chunk ahead:
// 711 -> 686 us (23,558 atoms, C = 128, l_max = 2), 27 -> 24 us (192 atoms,
// C = 64, l_max = 1). Measured and slower there: rows staged by bulk copies two
// visits ahead 779 us, two warps of 64 channels per atom 720 us, prefetches
// into L1 733 us; with every row in L1 it would take 594 us.
//
// Shared memory per block (15.3 KB at C = 128, l_max = 2): gA_a, 32 edge
// records of packs (f_c B_k, Y_lm, the r-derivative of f_c B_k), directions
// (n, 1/r) and neighbour indices, and the lanes' shares of the force of FT
// pairs (transposed so that four lanes add up each pair).
constexpr int FT = 8;   // pairs per force reduction

template <int C, int LMAX, int K>
struct BwdSmem {
    static constexpr int NL = LMAX + 1, NLM = NL * NL, CPW = C / 32;
    using T = typename Pack<CPW>::T;
    static constexpr int NP = Pack<CPW>::NP;
    static constexpr int V4 = 16 / sizeof(T);                       // packs per 16-byte word
    static constexpr int KY = (K + NLM + V4 - 1) / V4 * V4;         // f_c B_k and Y_lm, padded
    static constexpr int RW = ((KY + K) / V4) | 1;                  // 16-byte words per record, odd: conflict-free
    float4 rec[32][RW];
    float4 dir[32];
    float ga[NLM * C];
    float f[3][FT][33];
    int j[32];
};

// Words [0, N) of a record as packs.
template <int N, class T>
__device__ __forceinline__ void ld_rec(const float4 *p, T *v) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const float4 t = p[q];
        if constexpr (std::is_same<T, float2>::value) {
            v[2 * q] = make_float2(t.x, t.y);
            v[2 * q + 1] = make_float2(t.z, t.w);
        } else {
            v[4 * q] = t.x;
            v[4 * q + 1] = t.y;
            v[4 * q + 2] = t.z;
            v[4 * q + 3] = t.w;
        }
    }
}

template <int C, int LMAX, int K, bool VIR>
__global__ void __launch_bounds__(32) k_mp_bwd(EdgeGeom g, LayerIO io) {
    dep_entry(gridDim.x <= kOneWave);
    using S = BwdSmem<C, LMAX, K>;
    using T = typename S::T;
    constexpr int NL = S::NL, NLM = S::NLM, CPW = S::CPW, NP = S::NP, PW = Pack<CPW>::W, V4 = S::V4, KY = S::KY;
    extern __shared__ __align__(16) unsigned char mp_smem[];
    S &sm = *reinterpret_cast<S *>(mp_smem);
    const int lane = threadIdx.x;
    const Row rw = load_row(g, blockIdx.x);
    if (*io.err) return;
    const int a = rw.i, beg = rw.beg, end = rw.end;
    const int co = lane * CPW;   // this lane's channels
    // the first candidates
    int cj = beg + lane < end ? __ldg(g.col + beg + lane) : -1;
    T W[NL][K][NP];
#pragma unroll
    for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int k = 0; k < K; ++k) ldp<CPW>(io.wrad + (l * K + k) * C + co, W[l][k]);
    T sa[NP], san[NP], gse[NP], gso[NP];   // s_a, -s_a; sender-role sums over even and odd l
    ldp<CPW>(io.s + (size_t)a * C + co, sa);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        san[p] = vneg(sa[p]);
        gse[p] = vdup<T>(0.f);
        gso[p] = vdup<T>(0.f);
    }
    float cx = 0.f, cy = 0.f, cz = 0.f;
    if (cj >= 0) {
        cx = __ldg(g.x + 3 * cj);
        cy = __ldg(g.x + 3 * cj + 1);
        cz = __ldg(g.x + 3 * cj + 2);
    }
#pragma unroll
    for (int lm = 0; lm < NLM; ++lm) {
        T t[NP];
        ldp<CPW>(io.gA + ((size_t)a * NLM + lm) * C + co, t);
        stp<CPW>(sm.ga + lm * C + co, t);
    }
    const AtomGeom ge = wrap_inverse(rw.a);
    const float rc2 = g.rc * g.rc;
    // a's side of its pairs, fixed point (on the lanes that add up a pair)
    long long oa[3] = {0, 0, 0}, ow = 0;
    bool bad = false;   // a pair term outside the fixed-point range (or not finite)
    __syncwarp();

    for (int base = beg; base < end; base += 32) {
        bool act = false;
        const int j = cj;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j >= 0) {
            d = edge_disp(ge, cx, cy, cz);
            act = d.w < rc2;
        }
        // lower neighbours (j < a) first, then the upper ones (the pairs this
        // warp owns): rows are ascending, so g_s_a takes its terms in row
        // order whatever the chunk boundaries (which move with the list's
        // skin entries)
        const bool up = act && j > a, lo = act && j < a;
        const unsigned mu = __ballot_sync(DMTS_FULL, up), ml = __ballot_sync(DMTS_FULL, lo);
        const int n_lo = __popc(ml), nt = n_lo + __popc(mu);
        const unsigned lt = (1u << lane) - 1u;
        const int pos = lo ? __popc(ml & lt) : n_lo + __popc(mu & lt);
        if (up || lo) sm.j[pos] = j;
        const int en = base + 32 + lane;
        cj = en < end ? __ldg(g.col + en) : -1;
        if (up || lo) {
            const float r = sqrtf(d.w), inv = 1.f / r;
            float du;
            const float fc = envelope(r * g.inv_rc, g.p, &du);
            const float dfc = du * g.inv_rc;
            float B[K], dB[K], Y[NLM];
            bessel<K, true>(r, g.inv_rc, g.bnorm, B, dB);
            const float nx = d.x * inv, ny = d.y * inv, nz = d.z * inv;
            sph<LMAX>(nx, ny, nz, Y);
            sm.dir[pos] = make_float4(nx, ny, nz, inv);
            float v[KY + K];
#pragma unroll
            for (int q = 0; q < KY + K; ++q) {
                if (q < K) v[q] = fc * B[q < K ? q : 0];
                else if (q < K + NLM) v[q] = Y[q < K + NLM ? (q >= K ? q - K : 0) : 0];
                else if (q >= KY) v[q] = dfc * B[q >= KY ? q - KY : 0] + fc * dB[q >= KY ? q - KY : 0];
                else v[q] = 0.f;
            }
#pragma unroll
            for (int q = 0; q < (KY + K) / V4; ++q)
                sm.rec[pos][q] = V4 == 2 ? make_float4(v[2 * q], v[2 * q], v[2 * q + 1], v[2 * q + 1])
                                         : make_float4(v[V4 * q], v[V4 * q + 1], v[V4 * q + V4 / 2], v[V4 * q + V4 - 1]);
        }
        if (cj >= 0) {
            cx = __ldg(g.x + 3 * cj);
            cy = __ldg(g.x + 3 * cj + 1);
            cz = __ldg(g.x + 3 * cj + 2);
        }
        __syncwarp();

        // lower neighbours: the sender-role gradient only
#pragma unroll 2
        for (int t = 0; t < n_lo; ++t) {
            const float *row = io.gA + (size_t)sm.j[t] * NLM * C + co;
            T b[KY];
            ld_rec<KY / V4>(sm.rec[t], b);
            T wl[NL][NP];
#pragma unroll
            for (int lm = 0; lm < NLM; ++lm) {
                const int l = lm == 0 ? 0 : (lm < 4 ? 1 : 2);
                T gj[NP];
                ldp<CPW>(row + lm * C, gj);
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    wl[l][p] = lm == l * l ? vmul(gj[p], b[K + lm]) : vfma(gj[p], b[K + lm], wl[l][p]);
            }
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    T s0 = vmul(W[l][0][p], b[0]), s2 = vmul(W[l][1][p], b[1]);
#pragma unroll
                    for (int k = 2; k < K; k += 2) {
                        s0 = vfma(W[l][k][p], b[k], s0);
                        s2 = vfma(W[l][k + 1][p], b[k + 1], s2);
                    }
                    const T R = vadd(s0, s2);
                    if (l & 1) gso[p] = vfma(R, wl[l][p], gso[p]);
                    else gse[p] = vfma(R, wl[l][p], gse[p]);
                }
        }
#pragma unroll 1   // (two pairs at a time: 779 us, the compiler runs out of registers)
        for (int t = n_lo; t < nt; ++t) {
            const int jt = sm.j[t];
            const float *row = io.gA + (size_t)jt * NLM * C + co;
            T b[KY + K];
            ld_rec<(KY + K) / V4>(sm.rec[t], b);
            T sj[NP], rho, beta[NLM];
            ldp<CPW>(io.s + (size_t)jt * C + co, sj);
            rho = vdup<T>(0.f);
            T R[NL][NP], Rp[NL][NP];
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    T s0 = vmul(W[l][0][p], b[0]), s1 = vmul(W[l][0][p], b[KY]), s2 = vmul(W[l][1][p], b[1]),
                      s3 = vmul(W[l][1][p], b[KY + 1]);
#pragma unroll
                    for (int k = 2; k < K; k += 2) {
                        s0 = vfma(W[l][k][p], b[k], s0);
                        s1 = vfma(W[l][k][p], b[KY + k], s1);
                        s2 = vfma(W[l][k + 1][p], b[k + 1], s2);
                        s3 = vfma(W[l][k + 1][p], b[KY + k + 1], s3);
                    }
                    R[l][p] = vadd(s0, s2);
                    Rp[l][p] = vadd(s1, s3);
                }
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                T tl[NP], wl[NP];
#pragma unroll
                for (int lm = l * l; lm < (l + 1) * (l + 1); ++lm) {
                    T gj[NP], ga[NP];
                    ldp<CPW>(row + lm * C, gj);
                    ldp_s<CPW>(sm.ga + lm * C + co, ga);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const T gam = vfma(ga[p], sj[p], vmul(gj[p], (l & 1) ? san[p] : sa[p]));
                        const T y = b[K + lm];
                        tl[p] = lm == l * l ? vmul(gam, y) : vfma(gam, y, tl[p]);
                        beta[lm] = p == 0 ? vmul(gam, R[l][p]) : vfma(gam, R[l][p], beta[lm]);
                        wl[p] = lm == l * l ? vmul(gj[p], y) : vfma(gj[p], y, wl[p]);
                    }
                }
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    rho = vfma(Rp[l][p], tl[p], rho);
                    if (l & 1) gso[p] = vfma(R[l][p], wl[p], gso[p]);
                    else gse[p] = vfma(R[l][p], wl[p], gse[p]);
                }
            }
            // this lane's share (its channels) of the pair's force on a:
            // dY_lm/dd = (G_lm - (G_lm . n) n) / r with G_lm = grad_n Y_lm
            const float4 n = sm.dir[t];
            float h = vsum(rho), ex = 0.f, ey = 0.f, ez = 0.f;
            if (LMAX >= 1) {
                const float s3 = 1.7320508075688772f;
                float gx = s3 * vsum(beta[LMAX >= 1 ? 1 : 0]), gy = s3 * vsum(beta[LMAX >= 1 ? 2 : 0]),
                      gz = s3 * vsum(beta[LMAX >= 1 ? 3 : 0]);
                if (LMAX >= 2) {
                    const float s15 = 3.872983346207417f, s5 = 2.23606797749979f;
                    const float b4 = s15 * vsum(beta[LMAX >= 2 ? 4 : 0]), b5 = s15 * vsum(beta[LMAX >= 2 ? 5 : 0]),
                                b6 = 3.f * s5 * vsum(beta[LMAX >= 2 ? 6 : 0]),
                                b7 = s15 * vsum(beta[LMAX >= 2 ? 7 : 0]), b8 = s15 * vsum(beta[LMAX >= 2 ? 8 : 0]);
                    gx = fmaf(n.y, b4, fmaf(n.z, b7, fmaf(n.x, b8, gx)));
                    gy = fmaf(n.x, b4, fmaf(n.z, b5, fmaf(-n.y, b8, gy)));
                    gz = fmaf(n.y, b5, fmaf(n.x, b7, fmaf(n.z, b6, gz)));
                }
                h = fmaf(-n.w, fmaf(gx, n.x, fmaf(gy, n.y, gz * n.z)), h);
                ex = gx * n.w;
                ey = gy * n.w;
                ez = gz * n.w;
            }
            const int u = (t - n_lo) & (FT - 1);
            sm.f[0][u][lane] = fmaf(h, n.x, ex);
            sm.f[1][u][lane] = fmaf(h, n.y, ey);
            sm.f[2][u][lane] = fmaf(h, n.z, ez);
            const int done = t + 1 - n_lo;
            if (((done & (FT - 1)) == 0 || t + 1 == nt)) {
                __syncwarp();   // the shares are written
                // pair t0 + u: lanes u, u + 8, .. add up eight lanes' shares each
                // (conflict-free: row stride 33), then lane u the four parts, in
                // a fixed order
                const int t0 = n_lo + ((done - 1) & ~(FT - 1));
                const int u = lane & (FT - 1), h = lane / FT;
                const bool own = t0 + u <= t;
                float px = 0.f, py = 0.f, pz = 0.f;
                if (own) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        px += sm.f[0][u][8 * h + q];
                        py += sm.f[1][u][8 * h + q];
                        pz += sm.f[2][u][8 * h + q];
                    }
                }
                px += __shfl_down_sync(DMTS_FULL, px, 16);
                py += __shfl_down_sync(DMTS_FULL, py, 16);
                pz += __shfl_down_sync(DMTS_FULL, pz, 16);
                px += __shfl_down_sync(DMTS_FULL, px, 8);
                py += __shfl_down_sync(DMTS_FULL, py, 8);
                pz += __shfl_down_sync(DMTS_FULL, pz, 8);
                if (own && h == 0) {
                    const int jt = sm.j[t0 + u];
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
                            const float4 n = sm.dir[t0 + u];
                            const float wv = 0.5f / n.w * (px * n.x + py * n.y + pz * n.z);
                            if (fix_ok(wv)) {
                                const long long qw = to_fix(wv);
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
    ldp<CPW>(io.gs_in + (size_t)a * C + co, gin);
#pragma unroll
    for (int p = 0; p < NP; ++p) gout[p] = vfma(vdup<T>(io.nu), vsub(gse[p], gso[p]), gin[p]);
    stp<CPW>(io.gs_out + (size_t)a * C + co, gout);
    if (io.gs_out_bf16) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int hh = 0; hh < PW; ++hh)
                st_split(io.gs_out_bf16, a, C, co + p * PW + hh, vget(gout[p], hh));
    }
}

// One thread per atom: the adjoint's fixed-point forces (and virial) -> fp32,
// the words cleared for the next evaluation (also after an aborted one).
__global__ void k_fix_convert(int n, unsigned long long *__restrict__ Ffix, float *__restrict__ F,
                              unsigned long long *__restrict__ Wfix, float *__restrict__ W) {
    dep_entry();
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
    launch_dep(k_fix_convert, (n + 255) / 256, 256, 0, st, n, Ffix, F, Wfix, W);
    count_launch();
}

// In the forward pass 128 channels are split over two blocks (64 per warp):
// half the registers, twice the warps in flight to hide the neighbour loads.
template <int C, int LMAX>
static void fwd_c(const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    constexpr int SP = C >= 128 ? 2 : 1;
    const int blocks = (g.n_atoms + MP_WARPS - 1) / MP_WARPS;
    launch_dep_if(blocks <= (int)kOneWave / MP_WARPS, k_mp_fwd<C, LMAX, 8, SP>, dim3(blocks, SP), MP_WARPS * 32, 0, st, g, io);
    count_launch();
}

template <int C, int LMAX, bool VIR>
static void bwd_launch(const EdgeGeom &g, const LayerIO &io, cudaStream_t st) {
    constexpr size_t smem = sizeof(BwdSmem<C, LMAX, 8>);
    static_assert(smem <= 48 * 1024, "shared memory without an opt-in");
    launch_dep_if(g.n_atoms <= (int)kOneWave, k_mp_bwd<C, LMAX, 8, VIR>, g.n_atoms, 32, smem, st, g, io);
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
// fp32 SIMT contraction (fp32 models of fewer than 128 channels, small
// gradients; the others: gemm_split.cu). A CTA computes a BM x BN tile; K is walked in chunks
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
    dep_entry();
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
    launch_dep(k_gemm_f32<BM, BN, TM, TN>, grid, (BM / TM) * (BN / TN), smem, st, M, N, K, Act, W, trans, N % 4 == 0 && epilogue_vectorizable(e), e);
    count_launch();
}

// K is a multiple of 4 and both operands are 16-byte aligned (every
// contraction of the models: rows of C, (l_max + 1) C or 2 H n_c floats).
void launch_gemm_f32(int M, int N, int K, const float *Act, const float *W, int trans, const Epi &e,
                     cudaStream_t st) {
    if (M == 0) return;
    const int n_sm = sm_count();
    // small tiles until the large ones give every SM two CTAs: at 4,000 rows
    // (N = K = 128) 10.4 us against 8.3 (plain) and 12.3 against 12.4 (SiLU
    // epilogue), at 192 rows 6.2 against 8.3, at 23,558 rows 41 against 27
    if ((long long)((M + 63) / 64) * ((N + 63) / 64) >= 2LL * n_sm) gemm_f32_launch<64, 64, 4, 4>(M, N, K, Act, W, trans, e, st);
    else gemm_f32_launch<16, 32, 2, 2>(M, N, K, Act, W, trans, e, st);
}

// -------------------------------------------------- per-replica FP64 sums
__global__ void k_replica_sum(const float *__restrict__ v, const int *__restrict__ rep_off,
                              double *__restrict__ out, int accumulate) {
    dep_entry();
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
    launch_dep(k_replica_sum, n_rep, 1024, 0, st, v, rep_off, out, accumulate);
    count_launch();
}

}  // namespace dmts
