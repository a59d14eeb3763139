// Node-level MLP contractions on the 5th-generation tensor cores:
// Out[M][N] = Act[M][K] x W^T with bf16 operands and an fp32 accumulator in
// tensor memory, followed by the same fused epilogues as the fp32 GEMM.
//
// One CTA (eight warps) computes a 128 x BN tile (BN a multiple of 16 that
// divides N, near 64). Warp 0 (one lane) streams K-chunks of 64 bf16 of the
// activation tile and of the weight tile into shared memory with TMA
// (128-byte swizzle), warp 1 (one lane) issues tcgen05.mma (M = 128, N = BN,
// K = 16 per instruction) into a TMEM accumulator, warp 2 owns the TMEM
// allocation; warps 0-3 read the accumulator back with tcgen05.ld (warp w
// reads rows 32w..32w+31) into shared memory and all eight warps apply the
// epilogue with coalesced accesses.
//
// Split-bf16 operands (common.cuh: rows of 2K holding hi | lo) are
// contracted in three segments of K-chunks into the same accumulator,
// hi*hi + lo*hi + hi*lo, which keeps about 16 significant bits of each
// operand while every MMA is a plain bf16 x bf16 -> fp32 instruction.
//
// Every wait on an mbarrier is bounded: on timeout the CTA records
// DMTS_E_TIMEOUT, waits (bounded) for the loads and MMAs it has issued,
// frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "epilogue.cuh"
#include "launch.cuh"
#include "mp.cuh"
#include "ptx.cuh"
#include "tc.cuh"

namespace dmts {

namespace {

constexpr int TC_M = 128;
constexpr int TC_K = 64;             // bf16 elements per 128-byte swizzled row
constexpr int TC_STAGES = 4;
constexpr int kBNTarget = 64;      // preferred column-tile width

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// K-chunk k of a contraction over nseg segments (nk chunks each): segment 0
// multiplies the hi parts of both operands, segment 1 the activation's lo
// part with the weight's hi part, segment 2 the activation's hi part with
// the weight's lo part; kofs is the column where the lo parts start.
__device__ __forceinline__ void chunk_coords(int k, int nk, int kofs, int &xa, int &xb) {
    const int seg = k / nk, kc = k - seg * nk;
    xa = kc * TC_K + (seg == 1 ? kofs : 0);
    xb = kc * TC_K + (seg == 2 ? kofs : 0);
}

__global__ void __launch_bounds__(256) k_gemm_tc(const __grid_constant__ CUtensorMap tmA,
                                                 const __grid_constant__ CUtensorMap tmB, int M, int N, int K,
                                                 int BN, int tmem_cols, int n_stages, int vec, int nseg, int kofs,
                                                 Epi e, int *err) {
    dep_entry();
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[TC_STAGES], bar_empty[TC_STAGES], bar_done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh, issued_sh, consumed_sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // column tiles in reverse order: the gA epilogue's highest-degree tiles
    // (5 loads and stores per element for l = 2) are scheduled first
    const int m0 = blockIdx.x * TC_M, n0 = (gridDim.y - 1 - blockIdx.y) * BN;
    const int nk = K / TC_K, nkt = nk * nseg;
    const uint32_t a_bytes = TC_M * TC_K * 2, b_bytes = (uint32_t)BN * TC_K * 2;
    const uint32_t stage_bytes = a_bytes + ((b_bytes + 1023u) & ~1023u);
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;   // 1024-byte aligned tiles

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_done), 1);
        abort_sh = 0;
        issued_sh = 0;
        consumed_sh = 0;
        mbar_init_fence();
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;

    if (warp == 0 && lane == 0) {
        // ---- TMA producer
        int k = 0;
        for (; k < nkt; ++k) {
            const int s = k % n_stages;
            if (k >= n_stages && !mbar_wait(smem_u32(&bar_empty[s]), ((k / n_stages) - 1) & 1)) {
                atomicExch(&abort_sh, 1);
                break;
            }
            int xa, xb;
            chunk_coords(k, nk, kofs, xa, xb);
            const uint32_t sa = base + s * stage_bytes, sb = sa + a_bytes;
            mbar_expect_tx(smem_u32(&bar_full[s]), a_bytes + b_bytes);
            tma_load_2d(sa, &tmA, xa, m0, smem_u32(&bar_full[s]));
            tma_load_2d(sb, &tmB, xb, n0, smem_u32(&bar_full[s]));
        }
        issued_sh = k;   // loads issued; read after the block-wide barrier below
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        const uint32_t idesc = idesc_bf16(TC_M, BN);
        int k = 0;
        for (; k < nkt; ++k) {
            const int s = k % n_stages;
            if (!mbar_wait(smem_u32(&bar_full[s]), (k / n_stages) & 1)) {
                atomicExch(&abort_sh, 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa = base + s * stage_bytes, sb = sa + a_bytes;
#pragma unroll
            for (int kk = 0; kk < TC_K / 16; ++kk)
                mma_f16kind(tmem, smem_desc(sa + kk * 32), smem_desc(sb + kk * 32), idesc, (k > 0 || kk > 0) ? 1u : 0u);
            mma_commit(smem_u32(&bar_empty[s]));
        }
        consumed_sh = k;   // stages whose loads landed
        // arrives once every MMA issued above has completed
        mma_commit(smem_u32(&bar_done));
    }
    __syncwarp();
    // ---- epilogue: wait for the accumulator, read it back, fused epilogue
    const bool done = mbar_wait(smem_u32(&bar_done), 0);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!__syncthreads_and(done ? 1 : 0) || abort_sh) {
        if (threadIdx.x == 0) {
            atomicCAS(err, 0, (int)DMTS_E_TIMEOUT);
            // Drain before tensor and shared memory are released: every load
            // issued but not consumed (at most one per stage, the producer
            // refills a stage only after its MMAs completed) must land, and
            // the MMAs issued must complete; each wait again bounded.
            for (int k = consumed_sh; k < issued_sh; ++k)
                mbar_wait(smem_u32(&bar_full[k % n_stages]), (k / n_stages) & 1);
            if (!done) mbar_wait(smem_u32(&bar_done), 0);
        }
    } else {
        // TMEM -> shared memory (the drained pipeline buffers): warps 0-3
        // each move their 32-lane quarter, one row per lane. Then all eight
        // warps walk the tile row-major, consecutive threads on consecutive
        // columns, so the epilogue's loads and stores are coalesced and many
        // warps hide their latency.
        const int ld = BN + 1;
        float *tile = reinterpret_cast<float *>(smem_raw + (base - smem_u32(smem_raw)));
        if (warp < 4) {
            float *wtile = tile + (size_t)warp * 32 * ld;
            const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
            for (int c = 0; c < BN; c += 16) {
                float v[16];
                tmem_ld16(trow + (uint32_t)c, v);
#pragma unroll
                for (int q = 0; q < 16; ++q) wtile[lane * ld + c + q] = v[q];
            }
        }
        __syncthreads();
        const int rows = min(TC_M, M - m0);
        if (vec) epilogue_tile_v4(e, N, rows, m0, n0, BN, tile, ld);
        else epilogue_tile(e, N, rows, m0, n0, BN, tile, ld);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
    }
}

// ------------------------------------------------------------------- host
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::mutex g_encode_mutex;

bool encode_fn() {
    std::lock_guard<std::mutex> lock(g_encode_mutex);
    if (g_encode) return true;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return false;
    g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    return true;
}

// 2-D bf16 tensor map over rows x cols (row-major), box of box_rows x 64.
bool make_map(CUtensorMap *map, const void *ptr, int rows, int cols, int box_rows) {
    if (!encode_fn()) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_K, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Validity of a bf16 tensor-core contraction shape.
bool gemm_tc_supported(int N, int K) { return K % TC_K == 0 && K > 0 && N % 16 == 0 && N > 0; }

int launch_gemm_tc(int M, int N, int K, const __nv_bfloat16 *Act, const __nv_bfloat16 *Wt, const Epi &e, int *err,
                   cudaStream_t st, int split, int nseg) {
    if (M == 0) return 0;
    if (!gemm_tc_supported(N, K)) return -1;
    if (!(nseg == 1 || (split && nseg == 3))) return -1;
    const int width = split ? 2 * K : K;   // physical row length of both operands
    if (((uintptr_t)Act & 15) || ((uintptr_t)Wt & 15)) return -2;
    // column tile: the multiple of 16 dividing N closest to kBNTarget (the
    // smaller on a tie). Narrow tiles give more CTAs per SM (a smaller
    // epilogue staging tile) and more CTAs per contraction, which the
    // latency-bound epilogues of these short-K contractions need.
    int BN = 0;
    for (int b = 16; b <= 256 && b <= N; b += 16)
        if (N % b == 0 && (BN == 0 || std::abs(b - kBNTarget) < std::abs(BN - kBNTarget))) BN = b;
    if (!BN) return -1;
    // a narrow contraction (one or two column tiles) halves its tiles while
    // the grid has fewer than two CTAs per SM: these launches are bound by
    // latency, not by the second read of the activation tile (from L2)
    const int n_sm = sm_count();
    const int row_tiles = (M + TC_M - 1) / TC_M;
    while (BN % 32 == 0 && (long long)row_tiles * (N / BN) < 2LL * n_sm) BN /= 2;
    int tmem_cols = 32;
    while (tmem_cols < BN) tmem_cols <<= 1;
    CUtensorMap ma, mb;
    if (!make_map(&ma, Act, M, width, TC_M) || !make_map(&mb, Wt, N, width, BN)) return -3;
    const uint32_t stage = TC_M * TC_K * 2 + ((BN * TC_K * 2 + 1023) & ~1023);
    const int n_stages = std::min(3, nseg * K / TC_K);
    const size_t tile = (size_t)TC_M * (BN + 1) * sizeof(float);   // epilogue staging
    const size_t smem = std::max((size_t)stage * n_stages, tile) + 1024;
    // per launch: the attribute belongs to the current device's context
    cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    const int vec = epilogue_vectorizable(e);
    dim3 grid((M + TC_M - 1) / TC_M, N / BN);
    launch_dep(k_gemm_tc, grid, 256, smem, st, ma, mb, M, N, K, BN, tmem_cols, n_stages, vec, nseg, K, e, err);
    count_launch();
    return 0;
}

}  // namespace dmts
