// Projection GEMM for the bf16 path (paper Sec. 3.1: q, k, v = x*Wq, x*Wk, x*Wv):
//     C_w[M, N] = A[M, K] * B_w[K, N] (+ R[M, N]),  w < nW,  bf16 row-major operands, fp32 accumulation in TMEM;
// the optional residual R is added in the epilogue (the output projection of the attention block).
//
// Persistent kernel over output tiles of 128 CTAS rows by BN columns (all weight matrices in one launch).  CTAS = 2: a
// cluster of two CTAs works on one tile with cta_group::2 MMAs; each CTA holds 128 rows of A and of the accumulator and
// one half of the B columns.  Per CTA, warp 0 streams operand tiles with TMA into a shared-memory ring, warp 1 (of the
// first CTA) issues the MMAs (A K-major, B in its natural row-major form = MN-major) into one of two accumulators in
// TMEM, the other warps drain the other accumulator: a warp takes 32 rows by 64 columns at a time (TMEM -> registers ->
// bf16 -> a swizzled buffer of its own -> TMA store), so that no warp waits for another and a tile's epilogue runs under
// the next tile's main loop.
//
// What bounds it: a CTA of its own needs 48 KB of operands per 64-deep k-step for a 128 x 256 tile and an SM takes about 64
// bytes per cycle from L2: 740 cycles measured for 512 cycles of MMA (1.56 PFLOP/s over the chip).  A pair shares B, 32 KB per
// CTA and k-step, and takes 650 (1.79 PFLOP/s); M = 8192, N = 3 x 768: K = 3072 84.7 us with lone CTAs, 78.2 with pairs.  About
// 12 us do not scale with K: launch, first operands from DRAM, last epilogue.
#include <stdio.h>

#include <mutex>

#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

// ---------------------------------------------------------------- tensor-map helper
namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
std::once_flag g_encode_once;
}  // namespace

namespace {
bool resolve_encode() {
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    });
    if (!g_encode) { set_error_text("cuTensorMapEncodeTiled entry point not available"); return false; }
    return true;
}
}  // namespace

bool make_tensor_map_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint64_t pitch_bytes,
                          uint32_t box_rows, uint32_t box_cols) {
    if (!resolve_encode()) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {pitch_bytes};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char msg[96];
        snprintf(msg, sizeof(msg), "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
        set_error_text(msg);
        return false;
    }
    return true;
}

bool make_tensor_map_bf16_4d(CUtensorMap* map, const void* base, uint64_t batch, uint64_t n, uint64_t heads, uint64_t d,
                             uint32_t box_rows) {
    if (!resolve_encode()) return false;
    cuuint64_t dims[4] = {d, heads, n, batch};
    cuuint64_t strides[3] = {d * 2, heads * d * 2, n * heads * d * 2};
    cuuint32_t box[4] = {64, 1, box_rows, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char msg[96];
        snprintf(msg, sizeof(msg), "cuTensorMapEncodeTiled (4-D) failed with CUresult %d", (int)r);
        set_error_text(msg);
        return false;
    }
    return true;
}

namespace {

constexpr int BM = 128, BK = 64;               // rows of a CTA, depth of a k-step
constexpr int A_BYTES = BM * BK * 2;           // 16 KB, K-major [128 x 64]
constexpr int B_SUB_BYTES = BK * 64 * 2;       // 8 KB, one [64 k-rows x 64 n] sub-tile
constexpr int C_BUF_BYTES = 32 * 64 * 2;       // one staging buffer: 32 rows x 64 columns, bf16

template <int CTAS, int BN>
struct GCfg {
    static constexpr int NSUB = BN / 64;                       // 64-column sub-tiles of C per tile
    static constexpr int BSUB = NSUB / CTAS;                   // 64-column sub-tiles of B that a CTA loads
    static constexpr int STAGE_BYTES = A_BYTES + BSUB * B_SUB_BYTES;
    static constexpr int EPI_WARPS = 4;                        // (eight: 0.8 us more per launch, nothing gained)
    static constexpr int STAGES = 192 * 1024 / STAGE_BYTES;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr int SMEM = STAGES * STAGE_BYTES + EPI_WARPS * 2 * C_BUF_BYTES + 1024;     // + slack for 1024-byte alignment
    static constexpr int TMEM_COLS = BN > 128 ? 512 : 256;     // two accumulators (an allocation is a power of two)
};

struct GemmMaps {
    CUtensorMap a;
    CUtensorMap b[3];
    CUtensorMap c[3];
};

struct TileCoord {
    int w, m0, n0;
};
// Tile t of the launch: column tiles fastest, then row tiles, then the weight matrix, so that CTAs
// working side by side share the A row panel in L2.
__device__ __forceinline__ TileCoord tile_coord(int t, int mt, int nt, int bm, int bn) {
    TileCoord c;
    c.n0 = (t % nt) * bn;
    const int r = t / nt;
    c.m0 = (r % mt) * bm;
    c.w = r / mt;
    return c;
}

template <int CTAS, int BN, bool RES>
__global__ void __launch_bounds__(GCfg<CTAS, BN>::THREADS, 1)
gemm_bf16_kernel(const __grid_constant__ GemmMaps maps, int M, int N, int K, int nW, const uint16_t* __restrict__ R,
                 DeviceCounters* dc) {
    using Cfg = GCfg<CTAS, BN>;
    constexpr int STAGES = Cfg::STAGES, STAGE_BYTES = Cfg::STAGE_BYTES, NSUB = Cfg::NSUB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* stage_out = smem + STAGES * STAGE_BYTES;
    __shared__ uint64_t full_bar[STAGES], empty_bar[STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = CTAS == 2 ? (int)cluster_ctarank() : 0;   // the first CTA of a pair issues its MMAs
    const int unit = blockIdx.x / CTAS, units = gridDim.x / CTAS;
    const int nk = (K + BK - 1) / BK;
    const int mt = (M + CTAS * BM - 1) / (CTAS * BM), nt = (N + BN - 1) / BN;
    const int ntiles = mt * nt * nW;

    // full_bar and acc_empty of the first CTA serve the pair; empty_bar and acc_full exist in both and are completed in
    // both by one commit
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], CTAS * Cfg::EPI_WARPS); }
        fence_mbar_init();
    }
    if (warp == 1) {
        if constexpr (CTAS == 2) { tmem_alloc_pair(&tmem_base_s, Cfg::TMEM_COLS); tmem_relinquish_pair(); }
        else { tmem_alloc(&tmem_base_s, Cfg::TMEM_COLS); tmem_relinquish(); }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CTAS == 2) cluster_sync();       // the partner's barriers are initialised
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;
    // (programmatic dependent launch: the set-up above overlaps the end of the kernel before this one; the kernel after
    // this one is let in when a CTA's tiles are done, see attn_persist_kernel)
    grid_dependency_wait();

    if (warp == 0 && lane == 0) {
        // ---- TMA producer: k-steps of all this CTA's tiles, numbered g = 0, 1, ... through the ring.  The two CTAs of a pair
        // fill their halves of a stage on their own; the first CTA's barrier collects the bytes of both.
        int g = 0;
        bool ok = true;
        for (int t = unit; t < ntiles && ok; t += units) {
            const TileCoord c = tile_coord(t, mt, nt, CTAS * BM, BN);
            const int m0 = c.m0 + rank * BM, n0 = c.n0 + rank * Cfg::BSUB * 64;
            for (int kt = 0; kt < nk; ++kt, ++g) {
                const int s = g % STAGES;
                if (g >= STAGES && !mbar_wait(&empty_bar[s], ((g / STAGES) - 1) & 1, abortp)) { ok = false; break; }
                uint8_t* sA = smem + s * STAGE_BYTES;
                uint8_t* sB = sA + A_BYTES;
                if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], CTAS * STAGE_BYTES);
                if constexpr (CTAS == 2) {
                    const uint32_t bar = cluster_map(&full_bar[s], 0);
                    tma_load_2d_pair(sA, &maps.a, bar, kt * BK, m0);
#pragma unroll
                    for (int u = 0; u < Cfg::BSUB; ++u)
                        tma_load_2d_pair(sB + u * B_SUB_BYTES, &maps.b[c.w], bar, n0 + 64 * u, kt * BK);
                } else {
                    tma_load_2d(sA, &maps.a, &full_bar[s], kt * BK, m0);
#pragma unroll
                    for (int u = 0; u < Cfg::BSUB; ++u)
                        tma_load_2d(sB + u * B_SUB_BYTES, &maps.b[c.w], &full_bar[s], n0 + 64 * u, kt * BK);
                }
            }
        }
        // Let copies already in flight land before the CTA goes away.  (A pair's copies are all seen by the first CTA's
        // barriers, and neither CTA leaves before the other.)
        if (*abortp && rank == 0) {
            for (int k = max(0, g - STAGES); k < g; ++k) mbar_wait_drain(&full_bar[k % STAGES], (k / STAGES) & 1);
        }
    } else if (warp == 1 && rank == 0 && elect_one()) {
        // ---- MMA issuer (one elected lane of the converged warp; `lane == 0` and this, projection alone, us: 8192 rows x 2304 columns,
        // K = 768 29.2 and 27.6, K = 3072 74.1 and 72.4, 1024 rows 12.7 and 10.8)
        const uint32_t idesc = umma_idesc_bf16(CTAS * BM, BN, UMMA_K_MAJOR, UMMA_MN_MAJOR);
        // descriptor low words of stage 0; a stage or k-step is a constant added to them (sm100.cuh)
        const uint32_t a_lo0 = umma_desc_lo_kmajor(smem_u32(smem));
        const uint32_t b_lo0 = umma_desc_lo_mnmajor(smem_u32(smem + A_BYTES), B_SUB_BYTES);
        unsigned long long macs = 0;
        int g = 0, i = 0;
        bool ok = true;
        for (int t = unit; t < ntiles && ok; t += units, ++i) {
            const int buf = i & 1;
            if (i >= 2) ok = mbar_wait(&acc_empty[buf], ((i >> 1) - 1) & 1, abortp);   // epilogue drained it
            if (!ok) break;
            tc_fence_after();
            const uint32_t acc = tmem + buf * BN;
            for (int kt = 0; kt < nk; ++kt, ++g) {
                const int s = g % STAGES;
                ok = mbar_wait(&full_bar[s], (g / STAGES) & 1, abortp);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_lo = a_lo0 + s * (STAGE_BYTES >> 4), b_lo = b_lo0 + s * (STAGE_BYTES >> 4);
                auto mma = [&](int k, uint32_t accumulate) {
                    const uint64_t a = umma_desc_join(a_lo + k * (32 >> 4), UMMA_DESC_HI_SW128);
                    const uint64_t b = umma_desc_join(b_lo + k * (2048 >> 4), UMMA_DESC_HI_SW128);
                    if constexpr (CTAS == 2) umma_ss_pair(acc, a, b, idesc, accumulate);
                    else umma_ss(acc, a, b, idesc, accumulate);
                };
                if (kt == 0) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) mma(k, k != 0);
                } else {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) mma(k, 1);
                }
                if constexpr (CTAS == 2) umma_commit_pair(&empty_bar[s]);
                else umma_commit(&empty_bar[s]);
            }
            if (!ok) break;
            if constexpr (CTAS == 2) umma_commit_pair(&acc_full[buf]);
            else umma_commit(&acc_full[buf]);
            const TileCoord c = tile_coord(t, mt, nt, CTAS * BM, BN);
            macs += (unsigned long long)min(CTAS * BM, M - c.m0) * min(BN, N - c.n0) * K;
        }
        if (macs) atomicAdd(&dc->proj_macs, macs);
    } else if (warp >= 2) {
        // ---- epilogue: warp q owns TMEM lanes 32q .. 32q+31 = output rows
        const int q = warp & 3;
        uint8_t* buffers = stage_out + (warp - 2) * 2 * C_BUF_BYTES;
        const uint32_t empty0 = CTAS == 2 ? cluster_map(&acc_empty[0], 0) : 0, empty1 = CTAS == 2 ? cluster_map(&acc_empty[1], 0) : 0;
        int i = 0, stores = 0;
        for (int t = unit; t < ntiles; t += units, ++i) {
            const int buf = i & 1;
            const TileCoord c = tile_coord(t, mt, nt, CTAS * BM, BN);
            const int row0 = c.m0 + rank * BM + 32 * q, row = row0 + lane;
            // residual input: C = A B + R, added in fp32 before the rounding to bf16 (R is [M, N] bf16, row-major).  The
            // row's part of R is read while the tile is still being computed: sub-tile by sub-tile behind the
            // accumulator it cost 6 us on 8192 x 768.
            uint4 x[RES ? NSUB : 1][8];
            if constexpr (RES) {
                const uint4* rp = reinterpret_cast<const uint4*>(R + (size_t)row * N + c.n0);
#pragma unroll
                for (int u = 0; u < NSUB; ++u)
#pragma unroll
                    for (int g = 0; g < 8; ++g) x[u][g] = row < M && c.n0 + 64 * u < N ? __ldg(rp + 8 * u + g) : make_uint4(0, 0, 0, 0);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (i >> 1) & 1, abortp))) break;
            tc_fence_after();
#pragma unroll(RES ? NSUB : 1)
            for (int u = 0; u < NSUB; ++u) {
                const int col = c.n0 + 64 * u;
                uint32_t r[2][32];
                const uint32_t src = tmem + (static_cast<uint32_t>(q * 32) << 16) + buf * BN + u * 64;
                tmem_ld32(src, r[0]);
                tmem_ld32(src + 32, r[1]);
                tc_wait_ld();
                if (u == NSUB - 1) {                    // the accumulator may be overwritten by tile i + 2
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (CTAS == 2) mbar_arrive_cluster(buf ? empty1 : empty0);
                        else mbar_arrive(&acc_empty[buf]);
                    }
                }
                if constexpr (RES) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        const uint32_t w[4] = {x[u][g].x, x[u][g].y, x[u][g].z, x[u][g].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            uint32_t* dst = &r[g >> 2][(g & 3) * 8 + 2 * e];
                            dst[0] = __float_as_uint(__uint_as_float(dst[0]) + __uint_as_float(w[e] << 16));
                            dst[1] = __float_as_uint(__uint_as_float(dst[1]) + __uint_as_float(w[e] & 0xffff0000u));
                        }
                    }
                }
                uint8_t* sub = buffers + (stores & 1) * C_BUF_BYTES;
                if (stores >= 2) {                      // the store before the last must have read this buffer
                    if (lane == 0) tma_store_wait_read_1();
                    __syncwarp();
                }
#pragma unroll
                for (int c0 = 0; c0 < 2; ++c0) {
#pragma unroll
                    for (int g = 0; g < 4; ++g) {  // four 16-byte chunks of 8 bf16
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(r[c0][g * 8 + 0]), __uint_as_float(r[c0][g * 8 + 1]));
                        v.y = pack_bf16x2(__uint_as_float(r[c0][g * 8 + 2]), __uint_as_float(r[c0][g * 8 + 3]));
                        v.z = pack_bf16x2(__uint_as_float(r[c0][g * 8 + 4]), __uint_as_float(r[c0][g * 8 + 5]));
                        v.w = pack_bf16x2(__uint_as_float(r[c0][g * 8 + 6]), __uint_as_float(r[c0][g * 8 + 7]));
                        *reinterpret_cast<uint4*>(sub + swz128_offset(lane, c0 * 4 + g)) = v;
                    }
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (col < N && row0 < M) tma_store_2d(&maps.c[c.w], sub, col, row0);
                    tma_store_commit();                // (an empty group when the sub-tile lies outside the matrix)
                }
                ++stores;
            }
        }
        if (warp == 2 && lane == 0) grid_launch_dependents();
        if (lane == 0) tma_store_wait_read();      // shared memory may be released; the writes complete on their own
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if constexpr (CTAS == 2) {
        __syncwarp();
        cluster_sync();                 // MMAs, arrivals and copies that involve the partner are over in both CTAs
        tc_fence_after();
        if (warp == 1) tmem_dealloc_pair(tmem, Cfg::TMEM_COLS);
    } else {
        if (warp == 1) tmem_dealloc(tmem, Cfg::TMEM_COLS);
    }
}

template <int CTAS, int BN, bool RES>
int launch_gemm_kernel(const void* A, const void* const Bw[3], void* const C[3], int nW, int M, int K, int N, const void* residual,
                int sm_count, DeviceCounters* dc, cudaStream_t stream) {
    using Cfg = GCfg<CTAS, BN>;
    static DeviceSetup setup;
    if (device_setup(&setup, [] {
            return cudaFuncSetAttribute(gemm_bf16_kernel<CTAS, BN, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<CTAS, BN>::SMEM);
        }, "gemm set-up") <= 0)
        return PSA_ERR_CUDA;
    GemmMaps maps;
    if (!make_tensor_map_bf16(&maps.a, A, M, K, (uint64_t)K * 2, BM, BK)) return PSA_ERR_CUDA;
    for (int w = 0; w < 3; ++w) {
        const int src = w < nW ? w : 0;
        if (!make_tensor_map_bf16(&maps.b[w], Bw[src], K, N, (uint64_t)N * 2, BK, 64)) return PSA_ERR_CUDA;
        if (!make_tensor_map_bf16(&maps.c[w], C[src], M, N, (uint64_t)N * 2, 32, 64)) return PSA_ERR_CUDA;
    }
    const int ntiles = ((M + CTAS * BM - 1) / (CTAS * BM)) * ((N + BN - 1) / BN) * nW;
    const int units = ntiles < sm_count / CTAS ? ntiles : sm_count / CTAS;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(units * CTAS);
    cfg.blockDim = dim3(Cfg::THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CTAS;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CTAS == 2 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_bf16_kernel<CTAS, BN, RES>, maps, M, N, K, nW, static_cast<const uint16_t*>(residual), dc);
    if (e != cudaSuccess) { set_cuda_error(e, "gemm_bf16_kernel launch"); return PSA_ERR_CUDA; }
    return PSA_OK;
}

template <int CTAS, int BN>
int launch_gemm(const void* A, const void* const Bw[3], void* const C[3], int nW, int M, int K, int N, const void* residual,
                int sm_count, DeviceCounters* dc, cudaStream_t stream) {
    return residual ? launch_gemm_kernel<CTAS, BN, true>(A, Bw, C, nW, M, K, N, residual, sm_count, dc, stream)
                    : launch_gemm_kernel<CTAS, BN, false>(A, Bw, C, nW, M, K, N, residual, sm_count, dc, stream);
}

}  // namespace

int bf16_project(const void* A, const void* const Bw[3], void* const C[3], int nW, int M, int K, int N,
                 const void* residual, DeviceCounters* dc, cudaStream_t stream) {
    static DeviceSetup setup;
    const int sms = device_setup(&setup, [] { return cudaSuccess; }, "gemm set-up");
    if (sms <= 0) return PSA_ERR_CUDA;
    switch (gemm_tile(M, K, N, nW, sms)) {
        case GemmTile::LONE_128: return launch_gemm<1, 128>(A, Bw, C, nW, M, K, N, residual, sms, dc, stream);
        case GemmTile::LONE_192: return launch_gemm<1, 192>(A, Bw, C, nW, M, K, N, residual, sms, dc, stream);
        case GemmTile::LONE_256: return launch_gemm<1, 256>(A, Bw, C, nW, M, K, N, residual, sms, dc, stream);
        default: return launch_gemm<2, 256>(A, Bw, C, nW, M, K, N, residual, sms, dc, stream);
    }
}

}  // namespace psa
