// Fused attention core of the bf16 path for head sizes 128 < d_k <= 256 (FULL and MASKED schemes): phases 1-3 of the
// paper (Eq. 1-3) per (batch, head) and 128-row query tile, never materialising the weight matrix, as ONE persistent
// kernel with a CTA per SM.
//
// A 256-column output accumulator leaves tensor memory room for two score buffers of one row tile (S0 S1 | O, 512
// columns), P over the first half of its S.  Per key block S = Q K^T (16 MMAs of 128 x 128 x 16), softmax, O += P V (8 MMAs
// of 128 x 256 x 16); S of the next block is issued ahead of PV, so that the tensor pipe works on it during the
// softmax, and PV runs under the softmax of the next block.  The masked scheme's blocks beyond the diagonal are
// absent from every loop here too, and only the block on the diagonal carries an element predicate.
//
// Operands: Q 64 KB, and K and V through one ring of four 32 KB slots in the order the MMAs use them -- a K tile as two
// halves of the head's columns, a V tile as two halves of its keys -- so that a slot is free again after 8 or 4 MMAs.
//
// What bounds it: 16 MMAs of 64 cycles and 8 of 128 are 2048 cycles per block, 128 KB of operands at an SM's 64 bytes per
// cycle from L2 as many; the issuing thread spends 100-130 more on each of six barriers and five commits (with slots of 16 KB, nine of
// them, it was slower: 76 -> 89 us); measured 3000 on long sequences (16 heads of n = 8192, d_k = 192, masked: 559 us as one CTA per
// tile with one K and one V stage, 379 now; 32 heads of n = 2048, d_k = 256, masked: 103, then 80 and 70,
// the same inputs call after call; with other inputs every time 83 and 80).
//
// CTA layout (320 threads): warp 0 = work list and TMA producer, warp 1 = MMA issuer, warps 2-9 = softmax and epilogue
// (a warp owns 16 rows, read in the quad layout of sm100.cuh).  The tensors' head size may be any multiple of 8 in (128,
// 256]: columns beyond d_k are zero-filled by the loads and dropped by the stores.
#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_softmax.cuh"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int WD = 256;                                  // padded head width
constexpr int W_SUB = WD / 64;                           // 64-column sub-tiles of a tile
constexpr int W_Q_BYTES = 128 * WD * 2;                  // the Q tile: 64 KB
constexpr int W_SLOT_BYTES = W_Q_BYTES / 2;              // half a K or V tile: 32 KB
constexpr int W_SLOTS = 4;
constexpr int W_WARPS = SOFTMAX_WARPS_PER_TILE;          // 8
constexpr int W_THREADS = 32 * (CTRL_WARPS + W_WARPS);
constexpr int W_STAGE_BYTES = 16 * 64 * 2;               // output staging: 16 rows x 64 columns, two buffers per warp
constexpr int W_SMEM = W_Q_BYTES + W_SLOTS * W_SLOT_BYTES + W_WARPS * 2 * W_STAGE_BYTES + 1024;
constexpr int W_TMEM_S = 0, W_TMEM_O = 256;
constexpr int W_ITEM_READERS = W_WARPS + 1;              // softmax warps, MMA issuer

struct WMaps {
    CUtensorMap q, k, v, o;      // boxes of 128 rows (q, k), 64 rows (v), 16 rows (o) by 64 columns
};

struct WBars {
    uint64_t item_full[2], item_empty[2];
    uint64_t q_full, q_empty, r_full[W_SLOTS], r_empty[W_SLOTS];
    uint64_t s_full[2], p_ready[2], o_done[2];
};

__global__ void __launch_bounds__(W_THREADS, 1)
attn_wide_kernel(const __grid_constant__ WMaps maps, int n, int d, int H, int nbh, int group, int nitems, int scheme, float sl2,
                 DeviceCounters* dc, unsigned int* cursor, DeviceCounters* dc_next) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;
    uint8_t* sR = sQ + W_Q_BYTES;
    uint8_t* sStage = sR + W_SLOTS * W_SLOT_BYTES;
    __shared__ WBars bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;
    __shared__ int item_ring[2];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int T = row_tiles(n);
    const bool masked = scheme == PSA_MASKED;
    // Items are numbered group of heads by group of heads, inside a group row tile by row tile; the masked scheme starts with
    // the last (longest) row tile, so that the short ones fill the end.  FULL takes head by head (lpt_group in psa_sched.h):
    // with all heads in one group 128 heads of n = 1024 read K and V eight times from DRAM.
    auto item_work = [&](int idx, int& It, int& bh) {
        const int g = idx / (group * T), first = g * group, size = min(group, nbh - first);
        const int off = idx - first * T, r = off / size;
        bh = first + off - r * size;
        It = masked ? T - 1 - r : r;
    };

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int t = 0; t < 2; ++t) {
            mbar_init(&bars.item_full[t], 1);
            mbar_init(&bars.item_empty[t], W_ITEM_READERS);
            mbar_init(&bars.s_full[t], 1);
            mbar_init(&bars.p_ready[t], W_WARPS);          // one arrival per softmax warp
            mbar_init(&bars.o_done[t], 1);
        }
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_empty, 1);
        for (int s = 0; s < W_SLOTS; ++s) { mbar_init(&bars.r_full[s], 1); mbar_init(&bars.r_empty[s], 1); }
        fence_mbar_init();
    }
    if (warp == 1) { tmem_alloc(&tmem_base_s, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;
    grid_dependency_wait();      // (programmatic dependent launch, as in attn_persist_kernel)
    // the counter block of the NEXT call on this workspace is cleared here, off that call's critical path
    if (threadIdx.x == 0 && blockIdx.x == 0 && dc_next) *dc_next = DeviceCounters{0, 0, 0, 0, 0, 0, 0};

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------------ work list and TMA producer
            uint32_t rc = 0, qc = 0;                     // ring slots and Q tiles requested so far
            bool ok = true;
            int idx = blockIdx.x;                        // the grid never exceeds the item count
            int b = 0, h = 0;
            auto slot = [&]() -> int {                   // next ring slot, free; -1 when the wait ran out
                const int s = rc % W_SLOTS;
                if (rc >= (uint32_t)W_SLOTS && !mbar_wait(&bars.r_empty[s], ((rc / W_SLOTS) - 1) & 1, abortp)) return -1;
                mbar_arrive_expect_tx(&bars.r_full[s], W_SLOT_BYTES);
                ++rc;
                return s;
            };
            auto load_k = [&](int j) -> bool {           // K_j as column halves
                for (int half = 0; half < 2; ++half) {
                    const int s = slot();
                    if (s < 0) return false;
                    for (int u = 0; u < 2; ++u)
                        tma_load_4d(sR + s * W_SLOT_BYTES + u * 16384, &maps.k, &bars.r_full[s], 128 * half + 64 * u, h, j * TILE, b);
                }
                return true;
            };
            auto load_v = [&](int j) -> bool {           // V_j as key halves
                for (int half = 0; half < 2; ++half) {
                    const int s = slot();
                    if (s < 0) return false;
                    for (int u = 0; u < W_SUB; ++u)
                        tma_load_4d(sR + s * W_SLOT_BYTES + u * 8192, &maps.v, &bars.r_full[s], 64 * u, h, j * TILE + 64 * half, b);
                }
                return true;
            };
            for (uint32_t it = 0; ok; ++it) {
                if (it >= 2) ok = mbar_wait(&bars.item_empty[it & 1], ((it >> 1) - 1) & 1, abortp);
                if (!ok) break;
                item_ring[it & 1] = idx < nitems ? idx : -1;
                mbar_arrive(&bars.item_full[it & 1]);
                if (idx >= nitems) break;
                int It, bh;
                item_work(idx, It, bh);
                b = bh / H; h = bh - b * H;
                const int nkv = kv_tiles(It, T, scheme);
                if (qc > 0) ok = mbar_wait(&bars.q_empty, (qc - 1) & 1, abortp);
                if (!ok) break;
                mbar_arrive_expect_tx(&bars.q_full, W_Q_BYTES);
                for (int u = 0; u < W_SUB; ++u) tma_load_4d(sQ + u * 16384, &maps.q, &bars.q_full, 64 * u, h, It * TILE, b);
                ++qc;
                ok = load_k(0);
                int next = 0;
                for (int j = 0; j < nkv && ok; ++j) {
                    if (j + 1 < nkv) ok = load_k(j + 1);
                    if (ok) ok = load_v(j);
                    if (j == 0) next = (int)gridDim.x + (int)atomicAdd(cursor, 1u);      // (behind the item's first loads)
                }
                idx = next;
            }
            if (*abortp) {      // let copies already issued land before shared memory is released
                if (qc > 0) mbar_wait_drain(&bars.q_full, (qc - 1) & 1);
                for (uint32_t c = rc > (uint32_t)W_SLOTS ? rc - W_SLOTS : 0; c < rc; ++c) mbar_wait_drain(&bars.r_full[c % W_SLOTS], (c / W_SLOTS) & 1);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ------------------------------------------------------------ MMA issuer
            // (`lane == 0` instead of an elected lane: 76 and 70 us at 32 heads of n = 2048, d_k = 256, masked, 213 and 193 at 64 heads of n =
            // 2048, d_k = 192, full.)
            // Order of an item: S_0, S_1, PV_0, S_2, PV_1, ...  S_{j+1} overwrites S_{j-1} and P_{j-1}, which PV_{j-1}, issued
            // before it, has read: the tensor pipe runs this thread's MMAs in order.
            const uint32_t idescS = umma_idesc_bf16(128, 128, UMMA_K_MAJOR, UMMA_K_MAJOR);
            const uint32_t idescO = umma_idesc_bf16(128, WD, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t q_lo = umma_desc_lo_kmajor(smem_u32(sQ)), k_lo = umma_desc_lo_kmajor(smem_u32(sR));
            const uint32_t v_lo = umma_desc_lo_mnmajor(smem_u32(sR), 8192);
            const uint32_t dO = tmem + W_TMEM_O;
            uint32_t rc = 0, sc = 0, pc = 0;             // ring slots, S and PV so far
            bool ok = true;
            auto issue_S = [&](bool last) -> bool {      // phase 1 (Eq. 1): S = Q K^T, 128 columns of the head per ring slot
                const uint32_t dS = tmem + W_TMEM_S + (sc & 1) * 128;
#pragma unroll
                for (int half = 0; half < 2; ++half, ++rc) {
                    if (!mbar_wait(&bars.r_full[rc % W_SLOTS], (rc / W_SLOTS) & 1, abortp)) return false;
                    tc_fence_after();
                    const uint32_t k = k_lo + (rc % W_SLOTS) * (W_SLOT_BYTES >> 4);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const uint32_t off = ((kk >> 2) * 16384 + (kk & 3) * 32) >> 4;
                        umma_ss(dS, umma_desc_join(q_lo + half * (32768 >> 4) + off, UMMA_DESC_HI_SW128), umma_desc_join(k + off, UMMA_DESC_HI_SW128),
                                idescS, half != 0 || kk != 0);
                    }
                    umma_commit(&bars.r_empty[rc % W_SLOTS]);
                }
                umma_commit(&bars.s_full[sc & 1]);
                if (last) umma_commit(&bars.q_empty);
                ++sc;
                return true;
            };
            for (uint32_t it = 0; ok; ++it) {
                ok = mbar_wait(&bars.item_full[it & 1], (it >> 1) & 1, abortp);
                if (!ok) break;
                const int idx = item_ring[it & 1];
                mbar_arrive(&bars.item_empty[it & 1]);
                if (idx < 0) break;
                int It, bh;
                item_work(idx, It, bh);
                const int nkv = kv_tiles(It, T, scheme);
                ok = mbar_wait(&bars.q_full, it & 1, abortp) && issue_S(nkv == 1);
                for (int j = 0; j < nkv && ok; ++j) {
                    if (j + 1 < nkv) ok = issue_S(j + 2 == nkv);
                    if (ok) ok = mbar_wait(&bars.p_ready[pc & 1], (pc >> 1) & 1, abortp);
                    if (!ok) break;
                    const uint32_t aP = tmem + W_TMEM_S + (pc & 1) * 128;
#pragma unroll
                    for (int half = 0; half < 2; ++half, ++rc) {     // phase 3 (Eq. 3): O (+)= P_j V_j, 64 keys per ring slot
                        ok = mbar_wait(&bars.r_full[rc % W_SLOTS], (rc / W_SLOTS) & 1, abortp);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t v = v_lo + (rc % W_SLOTS) * (W_SLOT_BYTES >> 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            umma_ts(dO, aP + half * 32 + kk * 8, umma_desc_join(v + kk * (2048 >> 4), UMMA_DESC_HI_SW128), idescO,
                                    (j != 0 || half != 0 || kk != 0) ? 1u : 0u);
                        umma_commit(&bars.r_empty[rc % W_SLOTS]);
                    }
                    if (!ok) break;
                    umma_commit(&bars.o_done[pc & 1]);
                    ++pc;
                }
            }
            const unsigned long long block_macs = (unsigned long long)TILE * TILE * WD;
            if (sc) atomicAdd(&dc->qk_macs, sc * block_macs);
            if (pc) {
                atomicAdd(&dc->pv_macs, pc * block_macs);
                atomicAdd(&dc->exps, pc * (unsigned long long)(TILE * TILE));
            }
        }
    } else {
        // ------------------------------------------------------------ softmax + epilogue
        const int wq = warp - CTRL_WARPS;                       // softmax warp 0-7
        const int q = warp & 3;                                 // TMEM lane quarter this warp may access
        const int row0 = q * 32 + (wq >> 2) * 16;               // first of the warp's 16 rows inside the tile
        const int rA = row0 + (lane >> 2), rB = rA + 8;         // this thread's rows
        const int cq = 2 * (lane & 3);                          // its first column inside every group of 8
        const uint32_t lane_off = static_cast<uint32_t>(row0) << 16;
        const uint32_t tO = tmem + W_TMEM_O + lane_off;
        uint8_t* stage = sStage + wq * 2 * W_STAGE_BYTES;
        uint32_t blk = 0;                                       // blocks so far, all items
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bars.item_full[it & 1], (it >> 1) & 1, abortp));
            if (!ok) break;
            const int idx = item_ring[it & 1];
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.item_empty[it & 1]);
            if (idx < 0) break;
            int It, bh;
            item_work(idx, It, bh);
            const int nkv = kv_tiles(It, T, scheme);
            float mA = -INFINITY, mB = -INFINITY, lA = 0.f, lB = 0.f;       // running maxima (log2 units) and row sums
            for (int j = 0; j < nkv; ++j, ++blk) {
                ok = __all_sync(0xffffffffu, mbar_wait(&bars.s_full[blk & 1], (blk >> 1) & 1, abortp));
                if (!ok) break;
                const uint32_t tS = tmem + W_TMEM_S + (blk & 1) * 128 + lane_off;
                const int nvalid = min(TILE, n - j * TILE);
                const bool on_diag = masked && (j == It);
                const bool diag = on_diag || nvalid < TILE;
                const int cbA = min(on_diag ? rA : TILE - 1, nvalid - 1);
                const int cbB = min(on_diag ? rB : TILE - 1, nvalid - 1);
                uint32_t s0[32], s1[32];
                tc_fence_after();
                tmem_ld_quad64(tS, s0);
                tmem_ld_quad64(tS + 64, s1);
                tc_wait_ld();
                if (diag) {
                    mask_quad64(s0, cq, cbA, cbB);
                    mask_quad64(s1, 64 + cq, cbA, cbB);
                }
                float bA = -INFINITY, bB = -INFINITY;
                max_quad64(s0, bA, bB);
                max_quad64(s1, bA, bB);
                bA = quad_max(bA) * sl2;
                bB = quad_max(bB) * sl2;
                float alphaA = 1.f, alphaB = 1.f;
                if (bA > mA + RESCALE_THRESHOLD) {   // also taken on the first block (m = -inf)
                    alphaA = ex2_mufu(mA - bA);
                    mA = bA;
                }
                if (bB > mB + RESCALE_THRESHOLD) {
                    alphaB = ex2_mufu(mB - bB);
                    mB = bB;
                }
                // P over this warp's rows of S, which are in registers
                float sumA = 0.f, sumB = 0.f;
                uint32_t pk[16];
                exp_quad64(s0, sl2, -mA, -mB, pk, sumA, sumB);
                tmem_st_quad32(tS, pk);
                exp_quad64(s1, sl2, -mA, -mB, pk, sumA, sumB);
                tmem_st_quad32(tS + 32, pk);
                lA = fmaf(lA, alphaA, sumA);
                lB = fmaf(lB, alphaB, sumB);
                if (j > 0 && __any_sync(0xffffffffu, alphaA != 1.f || alphaB != 1.f)) {   // rare: a row maximum grew by > 2^8
                    const int nA = __popc(__ballot_sync(0xffffffffu, (lane & 3) == 0 && alphaA != 1.f));
                    const int nB = __popc(__ballot_sync(0xffffffffu, (lane & 3) == 0 && alphaB != 1.f));
                    if (lane == 0) atomicAdd(&dc->rescales, (unsigned long long)(nA + nB));
                    // O is at rest once the PV before this block's has committed
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars.o_done[(blk - 1) & 1], ((blk - 1) >> 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < WD / 64; ++c) {
                        uint32_t v[32];
                        tmem_ld_quad64(tO + 64 * c, v);
                        tc_wait_ld();
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            v[4 * g] = __float_as_uint(__uint_as_float(v[4 * g]) * alphaA);
                            v[4 * g + 1] = __float_as_uint(__uint_as_float(v[4 * g + 1]) * alphaA);
                            v[4 * g + 2] = __float_as_uint(__uint_as_float(v[4 * g + 2]) * alphaB);
                            v[4 * g + 3] = __float_as_uint(__uint_as_float(v[4 * g + 3]) * alphaB);
                        }
                        tmem_st_quad64(tO + 64 * c, v);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.p_ready[blk & 1]);
            }
            if (!ok) break;
            ok = __all_sync(0xffffffffu, mbar_wait(&bars.o_done[(blk - 1) & 1], ((blk - 1) >> 1) & 1, abortp));
            if (!ok) break;
            // ---- epilogue: y = O / l (the division of Eq. 2, applied once per output row), bf16, 64 columns at a time.  (The
            // next write to O, PV_0 of the next item, waits for that item's first P from every warp.)
            tc_fence_after();
            const int b = bh / H, h = bh - b * H;
            const float invA = 1.f / quad_sum(lA), invB = 1.f / quad_sum(lB);
#pragma unroll 1
            for (int u = 0; u < W_SUB; ++u) {
                uint32_t v[32];
                tmem_ld_quad64(tO + 64 * u, v);
                tc_wait_ld();
                uint8_t* sub = stage + (u & 1) * W_STAGE_BYTES;
                if (lane == 0) tma_store_wait_read_1();         // the store before the last must have read this buffer
                __syncwarp();
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const uint32_t a = pack_bf16x2(__uint_as_float(v[4 * g]) * invA, __uint_as_float(v[4 * g + 1]) * invA);
                    const uint32_t bb = pack_bf16x2(__uint_as_float(v[4 * g + 2]) * invB, __uint_as_float(v[4 * g + 3]) * invB);
                    *reinterpret_cast<uint32_t*>(sub + swz128_offset(lane >> 2, g) + 2 * cq) = a;
                    *reinterpret_cast<uint32_t*>(sub + swz128_offset((lane >> 2) + 8, g) + 2 * cq) = bb;
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (64 * u < d) tma_store_4d(&maps.o, sub, 64 * u, h, It * TILE + row0, b);
                    tma_store_commit();                         // (an empty group for a sub-tile wholly beyond the head's columns)
                }
            }
            tc_fence_before();
        }
        if (wq == 0 && lane == 0) grid_launch_dependents();
        if (lane == 0) tma_store_wait_read();    // shared memory may be released; the writes complete on their own
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace

// FULL and MASKED schemes for 128 < d <= 256 (d a multiple of 8).  `*cursor` must be zero when the kernel starts.
int bf16_attention_wide(const void* Q, const void* K, const void* V, void* out, int B, int H, int n, int d, float scale,
                        int scheme, DeviceCounters* dc, unsigned int* cursor, DeviceCounters* dc_next, cudaStream_t stream) {
    if (d <= 128 || d > WD || d % 8) return PSA_ERR_UNSUPPORTED;
    static DeviceSetup setup;
    const int sm_count = device_setup(&setup, [] {
        return cudaFuncSetAttribute(attn_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, W_SMEM);
    }, "wide attention kernel set-up");
    if (sm_count <= 0) return PSA_ERR_CUDA;
    WMaps maps;
    if (!make_tensor_map_bf16_4d(&maps.q, Q, B, n, H, d, 128) || !make_tensor_map_bf16_4d(&maps.k, K, B, n, H, d, 128) ||
        !make_tensor_map_bf16_4d(&maps.v, V, B, n, H, d, 64) || !make_tensor_map_bf16_4d(&maps.o, out, B, n, H, d, 16))
        return PSA_ERR_CUDA;
    const long long items = (long long)B * H * row_tiles(n);
    if (items > 0x7fffffffLL - 2 * sm_count) return PSA_ERR_SHAPE;       // (the work counter runs past the list)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((int)(items < sm_count ? items : sm_count));
    cfg.blockDim = dim3(W_THREADS);
    cfg.dynamicSmemBytes = W_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, attn_wide_kernel, maps, n, d, H, B * H, lpt_group(scheme, B * H, n, d), (int)items, scheme, scale * LOG2E, dc,
                                             cursor, dc_next);
    if (e != cudaSuccess) { set_cuda_error(e, "attn_wide_kernel launch"); return PSA_ERR_CUDA; }
    return PSA_OK;
}

}  // namespace psa
