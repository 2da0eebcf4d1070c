// Attention of the symmetric scheme (paper Sec. 4) with the weights themselves handed on, in bf16.
//
// With query = key = value = X the matrix of scores is symmetric, and so are the weights as long as every row has the same
// shift c: E_ij = exp(w'_ij - c) = E_ji.  Here c = 0, the literal form of the paper's Eq. 2: a row's largest weight is at least
// E_ii = exp(|x_i|^2 / sqrt d) >= 1, so nothing that matters underflows, and a bf16 weight has the same relative precision
// whatever its size.  What can happen is an overflow, and by Cauchy-Schwarz (w'_ij <= max(w'_ii, w'_jj)) the diagonal blocks
// show it: a head with a sum of weights beyond 2^100, or not a number, is given up, and sym_attn_kernel (psa_attn.cu),
// launched behind this one, works it off with running maxima; its other items are skipped here.
//
// So a block (I, J), J < I, is computed once, exponentiated once, used for O_I += E X_J from tensor memory and handed on
// through the scratch, 32 KB of bf16 in the layout of an operand, for O_J += E^T X_I, where the tensor core reads it transposed
// (an MN-major A operand) and no thread touches it.  The row sums of E^T are its column sums, which travel with it in fp32.
//
// Persistent, a CTA per SM; a CTA takes a whole head and works on its row tiles from the last to the first, so that what a tile wants
// handed on has been handed on by the same CTA.  A tile's blocks (I, I), (I, 0) .. (I, I - 1) are computed by one set of warps and
// its handed-on blocks (J, I), J > I, are taken up by another into the same accumulator while the next tile is being computed:
//   warp 0   work list, X tiles              warp 3   handed-on blocks with their X tiles, 64 keys at a time
//   warp 1   issues S = X_I X_J^T            warp 4   issues O += E^T X
//   warp 2   issues O += E X_J               warp 5   announces blocks handed on
//   warps 6-21   exponentials, in two groups that take blocks in turn (a warp owns 16 rows, quad layout of sm100.cuh)
//   warps 22-25  output rows
// Tensor memory: S0 S1 (E over its first half) | two accumulators.  The scratch is a ring of heads, some more than CTAs.
//
// Measured (1024 heads of n = 1024; us, handing on scores / weights): d = 128 1005 / 696, d = 32 862 / 552; 1024 heads of n = 512, d = 64
// 248 / 169, of n = 384 158 / 116; 256 heads of n = 2000, d = 64 872 / 703.  What bounds it: blocks, X tiles and the scratch move at 5.5 TB/s
// between L2 and the SMs, a head's 4 MB (n = 1024) being nobody else's.  Tried: the tiles of a head on different CTAs (they wait for one
// another in convoys, 1017 at d = 128), the tiles of two heads in turn (755; the ring is twice as large), handed-on lines discarded after use
// (no difference), sums added up lane by lane instead of by the warp's matrix instruction (25 more).
//
// The row sums are those of the weights as they were rounded: a row whose own weight is nearly all of it (the usual case here) then
// returns its own vector, whatever that weight was rounded to.
#include <algorithm>

#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_softmax.cuh"
#include "psa_sym.h"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int SH_GROUPS = 2, SH_GROUP_WARPS = 8, SH_SOFTMAX = SH_GROUPS * SH_GROUP_WARPS, SH_OUT_WARPS = 4;
constexpr int SH_FIRST_SOFTMAX = 6, SH_FIRST_OUT = SH_FIRST_SOFTMAX + SH_SOFTMAX;
constexpr int SH_THREADS = 32 * (SH_FIRST_OUT + SH_OUT_WARPS);      // 832
constexpr int SH_RING = 4;                                          // items between the first and the last role
constexpr int SH_READERS = 5 + SH_SOFTMAX + SH_OUT_WARPS;
constexpr int SH_STAGE_BYTES = 16 * 64 * 2;                         // a softmax warp's buffer for weights on their way out
constexpr int SH_E_HALF = SYM_E_BYTES / 2;                          // 64 keys of a handed-on block
constexpr float SH_LIMIT = 1.2676506e30f;                           // 2^100

struct ShBars {
    uint64_t item_full[SH_RING], item_empty[SH_RING], sums_here[SH_RING];
    uint64_t q_full, q_empty, x_full[4], x_empty[4], r_full[3], r_empty[3];
    uint64_t s_full[2], p_ready[2], o_done[2], a_done[2], b_done[2], l_ready[2], o_free[2];
};

template <int D>
struct ShCfg {
    static constexpr int SUB = D / 64;
    static constexpr int TILE_BYTES = 128 * D * 2;
    static constexpr int XST = D == 128 ? 3 : 4;                    // X tiles: two with scores ahead of their weights, one arriving
    static constexpr int RST = D == 128 ? 2 : 3;                    // half blocks handed on, with their X rows
    static constexpr int R_BYTES = SH_E_HALF + TILE_BYTES / 2;
    static constexpr int OFF_X = TILE_BYTES;
    static constexpr int OFF_R = OFF_X + XST * TILE_BYTES;
    static constexpr int OFF_STAGE = OFF_R + RST * R_BYTES;
    static constexpr int OFF_SUMS = OFF_STAGE + SH_SOFTMAX * SH_STAGE_BYTES;
    static constexpr int OFF_BARS = OFF_SUMS + 2 * SH_GROUPS * 128 * 4;
    static constexpr int OFF_MISC = OFF_BARS + (int)sizeof(ShBars);
    static constexpr int SMEM = OFF_MISC + 4 * (2 + SH_RING + SH_SOFTMAX);
    static constexpr int TMEM_O = 256;
};
static_assert(ShCfg<128>::SMEM <= 227 * 1024, "shared memory");

struct ShMaps {
    CUtensorMap x, xh;     // X as [batch, n, heads, d] bf16, boxes of 128 and of 64 rows x 64 columns
};

// Four 8 x 8 matrices of 16-bit elements, quad layout <-> rows of 16 bytes in shared memory (and back, transposed); lane l gives the
// address of row l % 8 of matrix l / 8.
__device__ __forceinline__ void stmatrix4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// Sums by the warp's matrix instruction: d += A 1 (row sums of a 16 x 16 piece of E in the quad layout: d[0] row A, d[2] row B) and
// d += 1 B (column sums of a 16 x 8 piece, transposed: d[0], d[1] of columns 2 (lane % 4) + 0, 1).
constexpr uint32_t SH_ONES = 0x3f803f80u;
__device__ __forceinline__ void mma_ones(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// heads: heads of this launch and of its header; slots: heads of blocks that the scratch behind the header holds.
template <int D>
__global__ void __launch_bounds__(SH_THREADS, 1)
sym_shared_kernel(const __grid_constant__ ShMaps maps, float* __restrict__ S, uint16_t* __restrict__ out, int n, int d, int H, int bh0, int heads,
                  int slots, float sl2, DeviceCounters* dc) {
    using Cfg = ShCfg<D>;
    constexpr int XST = Cfg::XST, RST = Cfg::RST;
    extern __shared__ __align__(1024) uint8_t sh_smem[];
    uint8_t* sQ = sh_smem;
    uint8_t* sX = sh_smem + Cfg::OFF_X;
    uint8_t* sR = sh_smem + Cfg::OFF_R;
    uint8_t* sStage = sh_smem + Cfg::OFF_STAGE;
    float* row_sums = reinterpret_cast<float*>(sh_smem + Cfg::OFF_SUMS);         // [item parity][group][row]
    ShBars& bars = *reinterpret_cast<ShBars*>(sh_smem + Cfg::OFF_BARS);
    int* misc = reinterpret_cast<int*>(sh_smem + Cfg::OFF_MISC);
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(misc);
    int* abort_s = misc + 1;
    int* item_ring = misc + 2;
    int* stored = misc + 2 + SH_RING;                                            // blocks whose weights a softmax warp has handed on

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int T = row_tiles(n);
    const SymHeader hd = sym_header(S, heads, T);
    uint8_t* blocks = reinterpret_cast<uint8_t*>(S) + sym_header_bytes(heads, T);
    const size_t head_bytes = sym_lower_blocks(T) * SYM_SHARED_BLOCK_BYTES;
    // item -> head and row tile, the last first
    auto item_work = [&](int idx, int& hl, int& It) {
        hl = idx / T;
        It = T - 1 - (idx - hl * T);
    };
    auto block_at = [&](int hl, int I, int J) { return blocks + (hl % slots) * head_bytes + sym_block_index(I, J) * SYM_SHARED_BLOCK_BYTES; };

    if (threadIdx.x == 0) {
        *abort_s = 0;
        for (int i = 0; i < SH_RING; ++i) { mbar_init(&bars.item_full[i], 1); mbar_init(&bars.item_empty[i], SH_READERS); mbar_init(&bars.sums_here[i], 1); }
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_empty, 2);                           // its last S, and its own values
        for (int i = 0; i < 4; ++i) { mbar_init(&bars.x_full[i], 1); mbar_init(&bars.x_empty[i], 1); }
        for (int i = 0; i < 3; ++i) { mbar_init(&bars.r_full[i], 1); mbar_init(&bars.r_empty[i], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.s_full[i], 1);
            mbar_init(&bars.p_ready[i], SH_GROUP_WARPS);       // one arrival per warp of the group
            mbar_init(&bars.o_done[i], 1);
            mbar_init(&bars.a_done[i], 1);
            mbar_init(&bars.b_done[i], 1);
            mbar_init(&bars.l_ready[i], SH_SOFTMAX);
            mbar_init(&bars.o_free[i], SH_OUT_WARPS);
        }
        fence_mbar_init();
    }
    if (threadIdx.x < SH_SOFTMAX) stored[threadIdx.x] = 0;
    if (warp == 1) { tmem_alloc(tmem_base_s, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_base_s;
    volatile int* abortp = abort_s;
    grid_dependency_wait();      // (programmatic dependent launch, as in attn_persist_kernel)

    // Entry `it` of the item ring, for the roles that take items one by one: its index, -1 at the end, -2 when the wait ran out.
    auto take_item = [&](uint32_t it) -> int {                 // (by whole warps)
        if (!__all_sync(0xffffffffu, mbar_wait(&bars.item_full[it % SH_RING], (it / SH_RING) & 1, abortp))) return -2;
        const int idx = item_ring[it % SH_RING];
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.item_empty[it % SH_RING]);
        return idx;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------------ work list, X tiles
            uint32_t xc = 0, qc = 0, it = 0;
            auto publish = [&](int idx) -> bool {
                if (it >= SH_RING && !mbar_wait(&bars.item_empty[it % SH_RING], (it / SH_RING - 1) & 1, abortp)) return false;
                item_ring[it % SH_RING] = idx;
                mbar_arrive(&bars.item_full[it % SH_RING]);
                ++it;
                return true;
            };
            auto tile = [&](int hl, int It) -> bool {
                if (ld_acquire(hd.bad + hl)) {      // a head given up: nothing more is done for it here
                    atomicAdd(hd.done + hl, SH_OUT_WARPS);
                    return true;
                }
                if (!publish(hl * T + T - 1 - It)) return false;
                const int bh = bh0 + hl, b = bh / H, h = bh - b * H;
                if (qc > 0 && !mbar_wait(&bars.q_empty, (qc - 1) & 1, abortp)) return false;
                mbar_arrive_expect_tx(&bars.q_full, Cfg::TILE_BYTES);
                for (int u = 0; u < Cfg::SUB; ++u) tma_load_4d(sQ + u * 16384, &maps.x, &bars.q_full, 64 * u, h, It * TILE, b);
                ++qc;
                for (int j = 0; j < It; ++j) {
                    const int s = xc % XST;
                    if (xc >= (uint32_t)XST && !mbar_wait(&bars.x_empty[s], ((xc / XST) - 1) & 1, abortp)) return false;
                    mbar_arrive_expect_tx(&bars.x_full[s], Cfg::TILE_BYTES);
                    for (int u = 0; u < Cfg::SUB; ++u)
                        tma_load_4d(sX + s * Cfg::TILE_BYTES + u * 16384, &maps.x, &bars.x_full[s], 64 * u, h, j * TILE, b);
                    ++xc;
                }
                return true;
            };
            bool ok = true;
            for (int head = atomicAdd(hd.work, 1); ok && head < heads; head = atomicAdd(hd.work, 1)) {
                // the blocks of the head `slots` heads before have been read
                if (head >= slots) ok = wait_at_least([&] { return ld_acquire(hd.done + head - slots); }, SH_OUT_WARPS * T, abortp);
                for (int It = T - 1; It >= 0 && ok; --It) ok = tile(head, It);
            }
            if (ok) publish(-1);
            if (*abortp) {  // let copies already issued land before shared memory is released
                if (qc > 0) mbar_wait_drain(&bars.q_full, (qc - 1) & 1);
                for (uint32_t c = xc > (uint32_t)XST ? xc - XST : 0; c < xc; ++c) mbar_wait_drain(&bars.x_full[c % XST], (c / XST) & 1);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ------------------------------------------------------------ issuer of S = X_I X_J^T, up to two blocks ahead of their use
            // (block 0 of an item is the diagonal one, whose keys and values are the row tile itself)
            const uint32_t idesc = umma_idesc_bf16(128, 128, UMMA_K_MAJOR, UMMA_K_MAJOR);
            const uint32_t q_lo = umma_desc_lo_kmajor(smem_u32(sQ)), k_lo = umma_desc_lo_kmajor(smem_u32(sX));
            uint32_t c = 0, xs = 0;
            bool ok = true;
            for (uint32_t it = 0; ok; ++it) {
                ok = mbar_wait(&bars.item_full[it % SH_RING], (it / SH_RING) & 1, abortp);
                if (!ok) break;
                const int idx = item_ring[it % SH_RING];
                mbar_arrive(&bars.item_empty[it % SH_RING]);
                if (idx < 0) break;
                int hl, It;
                item_work(idx, hl, It);
                ok = mbar_wait(&bars.q_full, it & 1, abortp);
                for (int b = 0; b <= It && ok; ++b, ++c) {
                    uint32_t k = q_lo;
                    if (b > 0) {
                        ok = mbar_wait(&bars.x_full[xs % XST], (xs / XST) & 1, abortp);
                        k = k_lo + (xs % XST) * (Cfg::TILE_BYTES >> 4);
                        ++xs;
                    }
                    if (ok && c >= 2) ok = mbar_wait(&bars.o_done[c & 1], ((c >> 1) - 1) & 1, abortp);      // the E in this buffer has been used
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = ((kk >> 2) * 16384 + (kk & 3) * 32) >> 4;
                        umma_ss(tmem + (c & 1) * 128, umma_desc_join(q_lo + off, UMMA_DESC_HI_SW128), umma_desc_join(k + off, UMMA_DESC_HI_SW128), idesc, kk != 0);
                    }
                    umma_commit(&bars.s_full[c & 1]);
                    if (b == It) {
                        umma_commit(&bars.q_empty);
                        atomicAdd(hd.qk_blocks + hl, It + 1);
                    }
                }
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            // ------------------------------------------------------------ issuer of O += E X_J
            const uint32_t idesc = umma_idesc_bf16(128, D, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t qv_lo = umma_desc_lo_mnmajor(smem_u32(sQ), 16384), v_lo = umma_desc_lo_mnmajor(smem_u32(sX), 16384);
            uint32_t c = 0, xp = 0;
            bool ok = true;
            for (uint32_t it = 0; ok; ++it) {
                ok = mbar_wait(&bars.item_full[it % SH_RING], (it / SH_RING) & 1, abortp);
                if (!ok) break;
                const int idx = item_ring[it % SH_RING];
                mbar_arrive(&bars.item_empty[it % SH_RING]);
                if (idx < 0) break;
                int hl, It;
                item_work(idx, hl, It);
                const uint32_t dO = tmem + Cfg::TMEM_O + (it & 1) * D;
                if (it >= 2) ok = mbar_wait(&bars.o_free[it & 1], ((it >> 1) - 1) & 1, abortp);
                for (int b = 0; b <= It && ok; ++b, ++c) {
                    ok = mbar_wait(&bars.p_ready[c & 1], (c >> 1) & 1, abortp);      // (its X tile has been there since its S)
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t v = b == 0 ? qv_lo : v_lo + (xp % XST) * (Cfg::TILE_BYTES >> 4), aP = tmem + (c & 1) * 128;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        umma_ts(dO, aP + kk * 8, umma_desc_join(v + kk * (2048 >> 4), UMMA_DESC_HI_SW128), idesc, (b != 0 || kk != 0) ? 1u : 0u);
                    umma_commit(&bars.o_done[c & 1]);
                    if (b == 0) umma_commit(&bars.q_empty);
                    else { umma_commit(&bars.x_empty[xp % XST]); ++xp; }
                    if (b == It) {
                        umma_commit(&bars.a_done[it & 1]);
                        atomicAdd(hd.pv_blocks + hl, It + 1);
                    }
                }
            }
        }
    } else if (warp == 3) {
        if (lane == 0) {
            // ------------------------------------------------------------ handed-on blocks and the X rows they go with
            uint32_t rc = 0;
            bool ok = true;
            for (uint32_t it = 0; ok; ++it) {
                ok = mbar_wait(&bars.item_full[it % SH_RING], (it / SH_RING) & 1, abortp);
                if (!ok) break;
                const int idx = item_ring[it % SH_RING];
                mbar_arrive(&bars.item_empty[it % SH_RING]);
                if (idx < 0) break;
                int hl, It;
                item_work(idx, hl, It);
                const int bh = bh0 + hl, b = bh / H, h = bh - b * H;
                if (It == T - 1) mbar_arrive(&bars.sums_here[it % SH_RING]);
                for (int J = T - 1; J > It && ok; --J) {
                    // Present once tile J has handed on more than It blocks.  They are announced tile by tile, so the flag of tile It +
                    // 2, which is looked at first, speaks for the tiles after it.  (A head given up hands on nothing any more: what is
                    // read then does not matter.)
                    if (J == T - 1 || J == It + 1) {
                        const int* flag = hd.flags + (size_t)hl * sym_flag_pitch(T) + min(J, It + (J == It + 1 ? 1 : 2));
                        ok = wait_at_least([&] {
                            const int v = ld_acquire(flag);
                            return v > It || !ld_acquire(hd.bad + hl) ? v : It + 1;
                        }, It + 1, abortp);
                        if (!ok) break;
                        if (J == It + 1) mbar_arrive(&bars.sums_here[it % SH_RING]);
                    }
                    asm volatile("fence.proxy.async;" ::: "memory");
                    const uint8_t* src = block_at(hl, J, It);
                    for (int half = 0; half < 2 && ok; ++half, ++rc) {
                        const int s = rc % RST;
                        if (rc >= (uint32_t)RST) ok = mbar_wait(&bars.r_empty[s], ((rc / RST) - 1) & 1, abortp);
                        if (!ok) break;
                        uint8_t* dst = sR + s * Cfg::R_BYTES;
                        mbar_arrive_expect_tx(&bars.r_full[s], Cfg::R_BYTES);
                        for (int u = 0; u < 2; ++u) bulk_load_1d(dst + u * (SH_E_HALF / 2), src + u * SH_E_HALF + half * (SH_E_HALF / 2), SH_E_HALF / 2, &bars.r_full[s]);
                        for (int u = 0; u < Cfg::SUB; ++u)
                            tma_load_4d(dst + SH_E_HALF + u * 8192, &maps.xh, &bars.r_full[s], 64 * u, h, J * TILE + 64 * half, b);
                    }
                }
            }
            if (*abortp)
                for (uint32_t c = rc > (uint32_t)RST ? rc - RST : 0; c < rc; ++c) mbar_wait_drain(&bars.r_full[c % RST], (c / RST) & 1);
        }
    } else if (warp == 4) {
        if (elect_one()) {
            // ------------------------------------------------------------ issuer of O += E^T X_J for the handed-on blocks
            const uint32_t idesc = umma_idesc_bf16(128, D, UMMA_MN_MAJOR, UMMA_MN_MAJOR);
            const uint32_t a_lo = umma_desc_lo_mnmajor(smem_u32(sR), SH_E_HALF / 2), b_lo = umma_desc_lo_mnmajor(smem_u32(sR + SH_E_HALF), 8192);
            uint32_t rc = 0;
            bool ok = true;
            for (uint32_t it = 0; ok; ++it) {
                ok = mbar_wait(&bars.item_full[it % SH_RING], (it / SH_RING) & 1, abortp);
                if (!ok) break;
                const int idx = item_ring[it % SH_RING];
                mbar_arrive(&bars.item_empty[it % SH_RING]);
                if (idx < 0) break;
                int hl, It;
                item_work(idx, hl, It);
                ok = mbar_wait(&bars.a_done[it & 1], (it >> 1) & 1, abortp);
                const uint32_t dO = tmem + Cfg::TMEM_O + (it & 1) * D;
                for (int t = 0; t < 2 * (T - 1 - It) && ok; ++t, ++rc) {
                    const uint32_t s = rc % RST;
                    ok = mbar_wait(&bars.r_full[s], (rc / RST) & 1, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = a_lo + s * (Cfg::R_BYTES >> 4), v = b_lo + s * (Cfg::R_BYTES >> 4);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        umma_ss(dO, umma_desc_join(a + kk * (2048 >> 4), UMMA_DESC_HI_SW128), umma_desc_join(v + kk * (2048 >> 4), UMMA_DESC_HI_SW128), idesc, 1);
                    umma_commit(&bars.r_empty[s]);
                }
                if (!ok) break;
                if (It < T - 1) {
                    umma_commit(&bars.b_done[it & 1]);
                    atomicAdd(hd.pv_blocks + hl, T - 1 - It);
                } else {
                    mbar_arrive(&bars.b_done[it & 1]);
                }
            }
        }
    } else if (warp == 5) {
        // ------------------------------------------------------------ announces blocks handed on
        // Lane w < 16 watches softmax warp w.  A block is complete when the eight warps of its group report their copies out as
        // complete; the fence orders those, observed through shared memory, before the flag.
        uint32_t cb = 0;                                        // number of the item's first block
        int sent[2] = {0, 0};                                   // blocks announced, by group
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            const int idx = take_item(it);
            if (idx < 0) break;
            int hl, It;
            item_work(idx, hl, It);
            int* flag = hd.flags + (size_t)hl * sym_flag_pitch(T) + It;
            for (int b = 1; b <= It; ++b) {
                const int g = (cb + b) & 1;
                const int target = ++sent[g];
                bool here = true;
                if (lane < SH_SOFTMAX && lane / SH_GROUP_WARPS == g) here = wait_at_least([&] { return ld_acquire_cta(stored + lane); }, target, abortp);
                ok = __all_sync(0xffffffffu, here);
                if (!ok) break;
                __syncwarp();
                if (lane == 0) {
                    __threadfence();
                    st_release(flag, b);
                }
            }
            cb += It + 1;
        }
    } else if (warp < SH_FIRST_OUT) {
        // ------------------------------------------------------------ exponentials
        const int sw = warp - SH_FIRST_SOFTMAX;                 // softmax warp 0-15
        const int grp = sw / SH_GROUP_WARPS, wq = sw % SH_GROUP_WARPS;
        const int q = warp & 3;                                 // TMEM lane quarter this warp may access
        const int kw = 2 * q + (wq >> 2);                       // its group of 16 rows inside the tile
        const int rA = 16 * kw + (lane >> 2);                   // this thread's rows: rA and rA + 8
        const int cq = 2 * (lane & 3);                          // its first column inside every group of 8
        const uint32_t tS = tmem + grp * 128 + (static_cast<uint32_t>(16 * kw) << 16);
        uint8_t* stage = sStage + sw * SH_STAGE_BYTES;
        // lane l addresses row l % 8 of matrix l / 8; matrices: rows A, rows B of column group g, then of group g + 1
        const uint32_t put = smem_u32(stage) + ((lane & 7) + (lane & 8)) * 128 + (((lane >> 4) ^ (lane & 7)) << 4);
        uint32_t c = 0;                                         // blocks so far, all items and both groups
        int nstored = 0;
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            const int idx = take_item(it);
            if (idx < 0) break;
            int hl, It;
            item_work(idx, hl, It);
            const int nvalid = min(TILE, n - It * TILE);        // rows of the tile (fewer than 128: the sequence's last, ragged tile)
            float lA = 0.f, lB = 0.f;
            for (int b = 0; b <= It; ++b, ++c) {
                if ((int)(c & 1) != grp) continue;
                ok = __all_sync(0xffffffffu, mbar_wait(&bars.s_full[grp], (c >> 1) & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                uint8_t* dst = block_at(hl, max(It, 1), max(b - 1, 0));
                const int last = b == 0 ? nvalid - 1 : TILE - 1;          // last key of the block
                const int cbA = rA < nvalid ? last : -1, cbB = rA + 8 < nvalid ? last : -1;
                float sumA = 0.f, sumB = 0.f;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t s[32], pk[16];
                    tmem_ld_quad64(tS + 64 * half, s);
                    tc_wait_ld();
                    if (nvalid < TILE) mask_quad64(s, 64 * half + cq, cbA, cbB);
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        pk[2 * g] = pack_bf16x2(ex2_mufu(__uint_as_float(s[4 * g]) * sl2), ex2_mufu(__uint_as_float(s[4 * g + 1]) * sl2));
                        pk[2 * g + 1] = pack_bf16x2(ex2_mufu(__uint_as_float(s[4 * g + 2]) * sl2), ex2_mufu(__uint_as_float(s[4 * g + 3]) * sl2));
                    }
                    tmem_st_quad32(tS + 32 * half, pk);         // E over this warp's rows of S, which are in registers
                    if (half == 1) {
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars.p_ready[grp]);
                    }
                    float rs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int g = 0; g < 8; g += 2) mma_ones(rs, pk[2 * g], pk[2 * g + 1], pk[2 * g + 2], pk[2 * g + 3], SH_ONES, SH_ONES);
                    sumA += rs[0];
                    sumB += rs[2];
                    if (b > 0) {
                        // ---- handed on: 16 rows x 64 columns through the warp's buffer, the column sums beside them
                        if (half == 1) {
                            if (lane == 0) tma_store_wait_read();         // the first half has left the buffer
                            __syncwarp();
                        }
#pragma unroll
                        for (int g = 0; g < 8; g += 2) stmatrix4(put ^ (g << 4), pk[2 * g], pk[2 * g + 1], pk[2 * g + 2], pk[2 * g + 3]);
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            bulk_store_1d(dst + half * SH_E_HALF + kw * SH_STAGE_BYTES, stage, SH_STAGE_BYTES);
                            tma_store_commit();
                        }
                        float2 cs = make_float2(0.f, 0.f);
#pragma unroll
                        for (int g = 0; g < 8; g += 2) {
                            uint32_t e[4];
                            ldmatrix4_trans(put ^ (g << 4), e);
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                float d[4] = {0.f, 0.f, 0.f, 0.f};
                                mma_ones(d, SH_ONES, SH_ONES, SH_ONES, SH_ONES, e[2 * u], e[2 * u + 1]);
                                if ((lane >> 2) == g + u) cs = make_float2(d[0], d[1]);
                            }
                        }
                        *reinterpret_cast<float2*>(dst + SYM_E_BYTES + 4 * (128 * kw + 64 * half + 8 * (lane >> 2) + cq)) = cs;
                    }
                }
                lA += sumA;
                lB += sumB;
                if (b > 0) {
                    __syncwarp();
                    if (lane == 0) { tma_store_wait_all(); st_release_cta(stored + sw, ++nstored); }
                } else if (__any_sync(0xffffffffu, !(sumA <= SH_LIMIT) || !(sumB <= SH_LIMIT))) {
                    if (lane == 0 && atomicExch(hd.bad + hl, 1) == 0) hd.list[atomicAdd(hd.given_up, 1)] = hl;
                }
            }
            if (!ok) break;
            if (__any_sync(0xffffffffu, !(lA <= SH_LIMIT) || !(lB <= SH_LIMIT))) {
                if (lane == 0 && atomicExch(hd.bad + hl, 1) == 0) hd.list[atomicAdd(hd.given_up, 1)] = hl;
            }
            // the sums of the item two before have been read
            if (it >= 2) ok = __all_sync(0xffffffffu, mbar_wait(&bars.o_free[it & 1], ((it >> 1) - 1) & 1, abortp));
            if (!ok) break;
            if ((lane & 3) == 0) {
                float* dst = row_sums + ((it & 1) * SH_GROUPS + grp) * 128 + rA;
                dst[0] = lA;
                dst[8] = lB;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.l_ready[it & 1]);
        }
        if (sw == 0 && lane == 0) grid_launch_dependents();
        if (lane == 0) tma_store_wait_read();
    } else {
        // ------------------------------------------------------------ output rows: y = O / l (the division of Eq. 2), bf16
        const int q = warp & 3, r = 32 * q + lane;              // TMEM lane quarter and row of this thread
        const bool wide = ((reinterpret_cast<uintptr_t>(out) | (uintptr_t)(2 * d)) & 31) == 0;
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            const int idx = take_item(it);
            if (idx < 0) break;
            int hl, It;
            item_work(idx, hl, It);
            const int par = it & 1;
            // the column sums of the handed-on blocks, while these are taken up: the accumulator is wanted again
            ok = __all_sync(0xffffffffu, mbar_wait(&bars.sums_here[it % SH_RING], (it / SH_RING) & 1, abortp));
            if (!ok) break;
            float l = 0.f;
#pragma unroll 4
            for (int J = It + 1; J < T; ++J) {
                const float* sums = reinterpret_cast<const float*>(block_at(hl, J, It) + SYM_E_BYTES) + r;
                float v[8];
#pragma unroll
                for (int w = 0; w < 8; ++w) v[w] = __ldcg(sums + 128 * w);
                l += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
            }
            ok = __all_sync(0xffffffffu, mbar_wait(&bars.l_ready[par], (it >> 1) & 1, abortp) && mbar_wait(&bars.b_done[par], (it >> 1) & 1, abortp));
            if (!ok) break;
            tc_fence_after();
            l += row_sums[par * SH_GROUPS * 128 + r] + row_sums[(par * SH_GROUPS + 1) * 128 + r];
            const float inv = 1.f / l;
            const int bh = bh0 + hl, bi = bh / H, h = bh - bi * H, row = It * TILE + r;
            uint16_t* y = out + (((size_t)bi * n + row) * H + h) * d;
#pragma unroll 1
            for (int c0 = 0; c0 < D; c0 += 32) {
                uint32_t v[32], w[16];
                tmem_ld32(tmem + Cfg::TMEM_O + par * D + c0 + (static_cast<uint32_t>(32 * q) << 16), v);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) w[e] = pack_bf16x2(__uint_as_float(v[2 * e]) * inv, __uint_as_float(v[2 * e + 1]) * inv);
                if (row < n) {
                    if (wide) {
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            if (c0 + 16 * e < d) st_global_32(y + c0 + 16 * e, w + 8 * e);
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (c0 + 8 * e < d) *reinterpret_cast<uint4*>(y + c0 + 8 * e) = make_uint4(w[4 * e], w[4 * e + 1], w[4 * e + 2], w[4 * e + 3]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars.o_free[par]);
                __threadfence();
                atomicAdd(hd.done + hl, 1);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_s) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// Places for a head's blocks: a quarter more than CTAs, so that a CTA does not wait for the last tile of another's head.
int sym_shared_slots(int heads, int T, size_t s_bytes, int sms) {
    const size_t fit = (s_bytes - sym_header_bytes(heads, T)) / (sym_lower_blocks(T) * SYM_SHARED_BLOCK_BYTES);
    return (int)std::min(fit, (size_t)std::min(heads, sms + sms / 4));
}

template <int D>
int launch(const void* X, void* out, float* S, size_t s_bytes, int heads, int bh0, int B, int H, int n, int d, float scale, DeviceCounters* dc,
           cudaStream_t stream) {
    using Cfg = ShCfg<D>;
    static DeviceSetup setup;
    const int sm_count = device_setup(&setup, [] {
        return cudaFuncSetAttribute(sym_shared_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, ShCfg<D>::SMEM);
    }, "cudaFuncSetAttribute(symmetric attention, weights handed on)");
    if (sm_count <= 0) return PSA_ERR_CUDA;
    const int T = row_tiles(n);
    ShMaps maps;
    if (!make_tensor_map_bf16_4d(&maps.x, X, B, n, H, d, 128) || !make_tensor_map_bf16_4d(&maps.xh, X, B, n, H, d, 64)) return PSA_ERR_CUDA;
    if ((long long)heads * T > 0x7fffffffLL) return PSA_ERR_SHAPE;
    const int grid = min(heads, sm_count), slots = sym_shared_slots(heads, T, s_bytes, sm_count);
    if (slots < 1) return PSA_ERR_WORKSPACE;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(SH_THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, sym_shared_kernel<D>, maps, S, static_cast<uint16_t*>(out), n, d, H, bh0, heads, slots,
                                             scale * LOG2E, dc);
    if (e != cudaSuccess) { set_cuda_error(e, "sym_shared_kernel launch"); return PSA_ERR_CUDA; }
    return PSA_OK;
}

}  // namespace

// Whether sym_shared_kernel is the better one.  A head per CTA leaves SMs idle where the heads are not many or just more than a multiple
// of them; with two tiles per head there is little to hand on (256 heads of n = 256, d = 128: 30 us, 37 here; 1024 heads 87 / 89), with
// three there is (256 heads of n = 384, d = 64 50 / 45); and the ring must have room for all CTAs' heads.
bool sym_shared_pays(int heads, int T, size_t s_bytes, int sms) {
    const int rounds = (heads + sms - 1) / sms;
    return T >= 3 && 3 * heads >= 2 * rounds * sms && sym_shared_slots(heads, T, s_bytes, sms) >= std::min(heads, sms);
}

int launch_sym_shared(const void* X, void* out, float* S, size_t s_bytes, int heads, int bh0, int B, int H, int n, int d, float scale,
                      DeviceCounters* dc, cudaStream_t stream) {
    if (d <= 64) return launch<64>(X, out, S, s_bytes, heads, bh0, B, H, n, d, scale, dc, stream);
    return launch<128>(X, out, S, s_bytes, heads, bh0, B, H, n, d, scale, dc, stream);
}

}  // namespace psa
