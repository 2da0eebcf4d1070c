// Attention core of the bf16 path: dispatch, and the kernel of the symmetric scheme (paper Sec. 4).
//
// With query = key = value = X the weight matrix before the softmax is symmetric, w'_ij = w'_ji (paper
// Eq. 4), and the paper computes one member of each pair and reuses it.  On this machine the reuse goes
// through memory, inside one persistent kernel: the CTA that works on 128-row tile I computes the blocks
// (I, J), J <= I, on the tensor core, uses them and hands those with J < I on through the scratch; for
// J > I it takes block (J, I) from there, transposed.  A block is written once and read once, and since a
// tile uses its computed blocks first and the handed-on ones after them, in the order of J, the tiles of a
// head run in step: block (J, I) is finished at step I of tile J and needed at step J of tile I, usually
// while it is still in L2.
//
// A work item is a row tile of one head.  Items are numbered group of heads by group of heads, inside a group
// the last tiles of all its heads first, and taken from a device counter in that order, so an item only ever
// waits for items that were taken before it: the oldest unfinished item waits for nobody.
//
// Roles of a CTA (352 threads): warp 0 takes items and loads operand tiles and handed-on blocks, warp 1 issues
// the MMAs, warps 2-9 do the softmax and the output (a warp owns 16 rows, quad layout of sm100.cuh), warp 10
// announces finished blocks to the other CTAs.  One row tile at a time, but with two score buffers and two
// weight buffers in tensor memory (S0 S1 | P0 P1 | O): S of the next block is there when the softmax of
// the current one ends, PV of a block runs under the softmax of the next, and the eight softmax warps drift
// apart by up to a block, which keeps the special-function pipe busy while some of them are at their loads.
//
// What bounds it: softmax (1024 cycles of exponentials per block) and, in step with it, the operands of one row
// tile per SM: 32 KB of X per block, 64 KB of scores stored or loaded for all but the diagonal one.  Measured
// (L2 flushed, B = 64, H = 16, n = 1024, d_k = 128): 1505 us as two kernels through 36 blocks written and 64 read
// per head, 917 us as one with 28 and 28.  An SM spends 4000 cycles per block; clock stamps of a softmax warp put
// 950 of them in the exponentials, 550 in the stores of computed blocks, 1000 in waits for handed-on ones.
//
// The fused persistent kernel of the FULL and MASKED schemes is in psa_attn_persist.cu.
#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_softmax.cuh"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int S_HALF_BYTES = S_BLOCK_BYTES / 2; // 64 of its rows = 64 key columns of the tile that reads it transposed
constexpr int SYM_WARPS = SOFTMAX_WARPS_PER_TILE;                    // 8
constexpr int SYM_PUBLISHER = CTRL_WARPS + SYM_WARPS;                // warp that announces finished blocks
constexpr int SYM_THREADS = 32 * (SYM_PUBLISHER + 1);                // 352
constexpr int SYM_ITEM_READERS = SYM_WARPS + 2;                      // softmax warps, MMA issuer, publisher

template <int D>
struct SymCfg {
    static constexpr int SUB = D / 64;                  // 64-column sub-tiles per 128-row tile of X
    static constexpr int TILE_BYTES = 128 * D * 2;      // one X tile (bf16)
    static constexpr int XST = D == 128 ? 3 : 4;        // X tiles in flight: PV of a block, S of the next, one loading (2: 5 % slower)
    static constexpr int MST = D == 128 ? 2 : 3;        // half blocks of handed-on scores in flight
    static constexpr int STAGE_BYTES = 16 * 64 * 4;     // a softmax warp's buffer for scores and outputs on their way out
    static constexpr int SMEM = (1 + XST) * TILE_BYTES + MST * S_HALF_BYTES + SYM_WARPS * STAGE_BYTES + 1024;
    static constexpr int TMEM_S = 0, TMEM_P = 256, TMEM_O = 384;
};

struct SymMaps {
    CUtensorMap x;     // X as [batch, n, heads, d] bf16, boxes of 128 rows x 64 columns
    CUtensorMap o;     // output, boxes of 16 rows
};

struct SymBars {
    uint64_t item_full[2], item_empty[2];
    uint64_t q_full, q_empty;
    uint64_t x_full[4], x_empty[4], m_full[4], m_empty[4];
    uint64_t s_full[2], s_free[2], p_ready[2], o_done[2];
};

// The scratch of a head is one 64 KB block per tile pair (I, J), J <= I, numbered I (I + 1) / 2 + J.  Diagonal blocks are
// never handed on; the place of block (0, 0) holds the head's flags instead: flag I = blocks that tile I has handed on.  The
// first head's place also holds, behind its T flags, the work counter of the launch.
__device__ __forceinline__ float* sym_head(float* Sg, int hl, int np) { return Sg + (size_t)hl * np * (S_BLOCK_BYTES / 4); }

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) { asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ int ld_acquire_cta(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta(int* p, int v) { asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory"); }

// Bounded wait until read() >= target.
template <class Read>
__device__ __forceinline__ bool wait_at_least(Read read, int target, volatile int* abort_flag) {
    if (read() >= target) return true;
    const uint64_t t0 = globaltimer_ns();
    while (read() < target) {
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > PSA_WAIT_LIMIT_NS) { *abort_flag = 1; return false; }
        __nanosleep(64);
    }
    return true;
}

template <int D>
__global__ void __launch_bounds__(SYM_THREADS, 1)
sym_attn_kernel(const __grid_constant__ SymMaps maps, float* __restrict__ Sg, int n, int H, int bh0, int heads, int group, float sl2,
                DeviceCounters* dc) {
    using Cfg = SymCfg<D>;
    constexpr int XST = Cfg::XST, MST = Cfg::MST;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;                                          // the row tile
    uint8_t* sX = sQ + Cfg::TILE_BYTES;                          // XST column tiles
    uint8_t* sM = sX + XST * Cfg::TILE_BYTES;                    // MST half blocks of handed-on scores
    uint8_t* sStage = sM + MST * S_HALF_BYTES;                   // output staging
    __shared__ SymBars bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;
    __shared__ int item_ring[2];
    __shared__ int stored[SYM_WARPS];                            // blocks whose scores a softmax warp has stored, all items

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int T = row_tiles(n);
    const int np = sym_pairs(T);
    const int nitems = heads * T;
    int* work_counter = reinterpret_cast<int*>(Sg) + T;
    // item -> head inside this pass and row tile: groups of heads, in a group the last tiles of all heads first
    auto item_work = [&](int idx, int& hl, int& It) {
        const int g = idx / (group * T), first = g * group, size = min(group, heads - first);
        const int off = idx - first * T, r = off / size;
        hl = first + off - r * size;
        It = T - 1 - r;
    };

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int t = 0; t < 2; ++t) {
            mbar_init(&bars.item_full[t], 1);
            mbar_init(&bars.item_empty[t], SYM_ITEM_READERS);
            mbar_init(&bars.s_full[t], 1);
            mbar_init(&bars.s_free[t], SYM_WARPS);               // one arrival per softmax warp
            mbar_init(&bars.p_ready[t], SYM_WARPS);
            mbar_init(&bars.o_done[t], 1);
        }
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_empty, 1);
        for (int s = 0; s < 4; ++s) {
            mbar_init(&bars.x_full[s], 1); mbar_init(&bars.x_empty[s], 1);
            mbar_init(&bars.m_full[s], 1); mbar_init(&bars.m_empty[s], SYM_WARPS);
        }
        fence_mbar_init();
    }
    if (threadIdx.x < SYM_WARPS) stored[threadIdx.x] = 0;
    if (warp == 1) { tmem_alloc(&tmem_base_s, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;
    grid_dependency_wait();      // (programmatic dependent launch, as in attn_persist_kernel)

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------------ work items, X tiles, handed-on score blocks
            uint32_t xc = 0, mc = 0, qc = 0;         // X tiles, half blocks and row tiles requested so far
            bool ok = true;
            int idx = atomicAdd(work_counter, 1);
            for (uint32_t it = 0; ok; ++it) {
                const int slot = it & 1;
                if (it >= 2) ok = mbar_wait(&bars.item_empty[slot], ((it >> 1) - 1) & 1, abortp);
                if (!ok) break;
                item_ring[slot] = idx < nitems ? idx : -1;
                mbar_arrive(&bars.item_full[slot]);
                if (idx >= nitems) break;
                int hl, It;
                item_work(idx, hl, It);
                const int bh = bh0 + hl, b = bh / H, h = bh - b * H;
                float* head = sym_head(Sg, hl, np);
                const int* flags = reinterpret_cast<const int*>(head);
                int next = 0;
                for (int j = 0; j < T && ok; ++j) {
                    const int s = xc % XST;
                    if (xc >= (uint32_t)XST) ok = mbar_wait(&bars.x_empty[s], ((xc / XST) - 1) & 1, abortp);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&bars.x_full[s], Cfg::TILE_BYTES);
                    for (int u = 0; u < Cfg::SUB; ++u)
                        tma_load_4d(sX + s * Cfg::TILE_BYTES + u * 16384, &maps.x, &bars.x_full[s], 64 * u, h, j * TILE, b);
                    ++xc;
                    if (j == 0) {
                        if (qc > 0) ok = mbar_wait(&bars.q_empty, (qc - 1) & 1, abortp);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&bars.q_full, Cfg::TILE_BYTES);
                        for (int u = 0; u < Cfg::SUB; ++u) tma_load_4d(sQ + u * 16384, &maps.x, &bars.q_full, 64 * u, h, It * TILE, b);
                        ++qc;
                    }
                    // the next item, as late as its answer's way allows: items then start in the order of their numbers
                    if (j == max(T - 3, 0)) next = atomicAdd(work_counter, 1);
                    if (j <= It) continue;
                    // block (j, It), handed on by the CTA that works on tile j: present once its flag counts past It.  The
                    // flag is an ordinary load, the copies below go through the asynchronous proxy.
                    ok = wait_at_least([&] { return ld_acquire(flags + j); }, It + 1, abortp);
                    if (!ok) break;
                    asm volatile("fence.proxy.async;" ::: "memory");
                    const float* src = head + (size_t)(j * (j + 1) / 2 + It) * (S_BLOCK_BYTES / 4);
                    for (int half = 0; half < 2 && ok; ++half) {
                        const int ms = mc % MST;
                        if (mc >= (uint32_t)MST) ok = mbar_wait(&bars.m_empty[ms], ((mc / MST) - 1) & 1, abortp);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&bars.m_full[ms], S_HALF_BYTES);
                        for (int u = 0; u < 2; ++u)
                            bulk_load_1d(sM + ms * S_HALF_BYTES + u * (S_HALF_BYTES / 2), src + half * (S_HALF_BYTES / 4) + u * (S_HALF_BYTES / 8),
                                         S_HALF_BYTES / 2, &bars.m_full[ms]);
                        ++mc;
                    }
                }
                idx = next;
            }
            if (*abortp) {  // let copies already issued land before shared memory is released
                if (qc > 0) mbar_wait_drain(&bars.q_full, (qc - 1) & 1);
                for (uint32_t c = xc > (uint32_t)XST ? xc - XST : 0; c < xc; ++c) mbar_wait_drain(&bars.x_full[c % XST], (c / XST) & 1);
                for (uint32_t c = mc > (uint32_t)MST ? mc - MST : 0; c < mc; ++c) mbar_wait_drain(&bars.m_full[c % MST], (c / MST) & 1);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ------------------------------------------------------------ MMA issuer
            // Per item S_0 .. S_It (phase 1, Eq. 1) and PV_0 .. PV_{T-1} (phase 3, Eq. 3), each S one block ahead of its PV;
            // the first S of the next item runs under the output of this one.
            const uint32_t idescS = umma_idesc_bf16(128, 128, UMMA_K_MAJOR, UMMA_K_MAJOR);
            const uint32_t idescO = umma_idesc_bf16(128, D, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t q_lo = umma_desc_lo_kmajor(smem_u32(sQ)), k_lo = umma_desc_lo_kmajor(smem_u32(sX));
            const uint32_t v_lo = umma_desc_lo_mnmajor(smem_u32(sX), 16384);
            uint32_t sc = 0, pc = 0, xbase = 0, it = 0;      // S and PV issued so far; ring position of the item's first X tile
            bool ok = true;
            auto take = [&]() -> int {                        // next item: index, -1 at the end, -2 when a wait ran out
                if (!mbar_wait(&bars.item_full[it & 1], (it >> 1) & 1, abortp)) return -2;
                const int idx = item_ring[it & 1];
                mbar_arrive(&bars.item_empty[it & 1]);
                ++it;
                return idx;
            };
            auto issue_S = [&](uint32_t xpos, bool first, bool last) -> bool {
                if (first && !mbar_wait(&bars.q_full, (it - 1) & 1, abortp)) return false;
                if (!mbar_wait(&bars.x_full[xpos % XST], (xpos / XST) & 1, abortp)) return false;
                if (sc >= 2 && !mbar_wait(&bars.s_free[sc & 1], ((sc >> 1) - 1) & 1, abortp)) return false;
                tc_fence_after();
                const uint32_t k = k_lo + (xpos % XST) * (Cfg::TILE_BYTES >> 4), dS = tmem + Cfg::TMEM_S + (sc & 1) * 128;
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off = ((kk >> 2) * 16384 + (kk & 3) * 32) >> 4;
                    umma_ss(dS, umma_desc_join(q_lo + off, UMMA_DESC_HI_SW128), umma_desc_join(k + off, UMMA_DESC_HI_SW128), idescS, kk != 0);
                }
                umma_commit(&bars.s_full[sc & 1]);
                if (last) umma_commit(&bars.q_empty);
                ++sc;
                return true;
            };
            int idx = take();
            int hl, It = 0;
            if (idx >= 0) item_work(idx, hl, It);
            if (idx >= 0) ok = issue_S(0, true, It == 0);
            while (idx >= 0 && ok) {
                int idx_next = -1, It_next = 0;
                for (int j = 0; j < T; ++j) {
                    if (j < It) ok = issue_S(xbase + j + 1, false, j + 1 == It);
                    const uint32_t xpos = xbase + j;
                    if (ok && j > It) ok = mbar_wait(&bars.x_full[xpos % XST], (xpos / XST) & 1, abortp);
                    if (ok) ok = mbar_wait(&bars.p_ready[pc & 1], (pc >> 1) & 1, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t v = v_lo + (xpos % XST) * (Cfg::TILE_BYTES >> 4);
                    const uint32_t aP = tmem + Cfg::TMEM_P + (pc & 1) * 64, dO = tmem + Cfg::TMEM_O;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        umma_ts(dO, aP + kk * 8, umma_desc_join(v + kk * (2048 >> 4), UMMA_DESC_HI_SW128), idescO, (j != 0 || kk != 0) ? 1u : 0u);
                    umma_commit(&bars.o_done[pc & 1]);
                    umma_commit(&bars.x_empty[xpos % XST]);
                    ++pc;
                }
                if (!ok) break;
                idx_next = take();
                if (idx_next == -2) break;
                if (idx_next >= 0) {
                    item_work(idx_next, hl, It_next);
                    ok = issue_S(xbase + T, true, It_next == 0);
                }
                xbase += T;
                idx = idx_next;
                It = It_next;
            }
            const unsigned long long block_macs = (unsigned long long)TILE * TILE * D;
            if (sc) atomicAdd(&dc->qk_macs, sc * block_macs);
            if (pc) {
                atomicAdd(&dc->pv_macs, pc * block_macs);
                atomicAdd(&dc->exps, pc * (unsigned long long)(TILE * TILE));
            }
        }
    } else if (warp == SYM_PUBLISHER) {
        // ------------------------------------------------------------ announces blocks handed on
        // Lane w < 8 watches softmax warp w.  A block is complete when all eight report their copies out as complete; the fence
        // orders those, observed through shared memory, before the flag.
        int done = 0;                                           // blocks announced in earlier items
        for (uint32_t it = 0;; ++it) {
            if (!__all_sync(0xffffffffu, mbar_wait(&bars.item_full[it & 1], (it >> 1) & 1, abortp))) break;
            const int idx = item_ring[it & 1];
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.item_empty[it & 1]);
            if (idx < 0) break;
            int hl, It;
                item_work(idx, hl, It);
            int* flag = reinterpret_cast<int*>(sym_head(Sg, hl, np)) + It;
            int sent = 0;
            bool ok = true;
            while (sent < It) {
                const int* mine = &stored[lane & (SYM_WARPS - 1)];
                ok = __all_sync(0xffffffffu, wait_at_least([&] { return ld_acquire_cta(mine); }, done + sent + 1, abortp));
                if (!ok) break;
                const int ready = __reduce_min_sync(0xffffffffu, ld_acquire_cta(mine)) - done;    // may have moved on
                sent = min(ready, It);
                __syncwarp();
                if (lane == 0) {
                    __threadfence();
                    st_release(flag, sent);
                }
            }
            if (!ok) break;
            done += It;
        }
    } else {
        // ------------------------------------------------------------ softmax + epilogue
        const int wq = warp - CTRL_WARPS;                       // softmax warp 0-7
        const int q = warp & 3;                                 // TMEM lane quarter this warp may access
        const int kw = 2 * q + (wq >> 2);                       // its group of 16 rows inside the tile
        const int row0 = 16 * kw;
        const int cq = 2 * (lane & 3);                          // the thread's first column inside every group of 8
        const uint32_t lane_off = static_cast<uint32_t>(row0) << 16;
        const uint32_t tO = tmem + Cfg::TMEM_O + lane_off;
        uint8_t* stage = sStage + wq * Cfg::STAGE_BYTES;
        // Place of a score in a handed-on block, in floats: [16-row group of the writer][column half][group of 8 columns]
        // [chunk][column parity][row A / B].  A writer thread stores its four scores of a column group as one 16-byte chunk;
        // element (r, c) is row c, key r of the reader, which takes keys r and r + 8 as 8 bytes.  With r2 r1 r0 the row and c1 c0
        // the column pair inside an 8 x 8 square, the chunk's number is (r2, r1, r2 ^ r0, r1 ^ c1, c0): the 8 lanes of a
        // writing phase and the 16 of a reading one then touch every bank once.
        const int put = 4 * ((lane & 1) | ((lane ^ (lane >> 2)) & 2) | ((lane ^ (lane >> 2)) & 4) | (lane & 24));
        const int get_chunk = ((lane >> 3) & 1) | (((lane ^ (lane >> 4)) & 1) << 1) | ((lane & 2) << 1) | ((lane & 1) << 3) | ((lane & 2) << 3);
        const int get = (kw >> 2) * 1024 + (kw & 3) * 256 + 2 * ((lane >> 2) & 1);
        const int get_even = get + 4 * get_chunk, get_odd = get + 4 * (get_chunk ^ 4);      // rows r with r0 = 0, 1
        uint32_t blk = 0, sc = 0, mc = 0;                       // blocks, computed blocks and half blocks so far, all items
        int nstored = 0;
        bool handed = false;                                    // the block before was handed on and not yet reported
        // Half a block's scores of this warp (16 rows, 64 columns) go out through its buffer as one bulk copy.  (Stored from the
        // registers they take the warps 1100 cycles per block, an SM's way out being 64 bytes wide.)
        auto hand_on = [&](const uint32_t (&s)[32], float* dst) {
            if (lane == 0) tma_store_wait_read();               // whatever used the buffer last
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 8; ++g)
                *reinterpret_cast<uint4*>(stage + 512 * g + 4 * put) = make_uint4(s[4 * g], s[4 * g + 2], s[4 * g + 1], s[4 * g + 3]);
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                bulk_store_1d(dst, stage, Cfg::STAGE_BYTES);
                tma_store_commit();
            }
        };
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bars.item_full[it & 1], (it >> 1) & 1, abortp));
            if (!ok) break;
            const int idx = item_ring[it & 1];
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.item_empty[it & 1]);
            if (idx < 0) break;
            int hl, It;
                item_work(idx, hl, It);
            float* own = sym_head(Sg, hl, np) + (size_t)(It * (It + 1) / 2) * (S_BLOCK_BYTES / 4) + kw * 2048;
            float mA = -INFINITY, mB = -INFINITY, lA = 0.f, lB = 0.f;       // running maxima (log2 units) and row sums
            for (int j = 0; j < T; ++j, ++blk) {
                uint32_t s0[32], s1[32];
                if (j <= It) {
                    // ---- a block computed here
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars.s_full[sc & 1], (sc >> 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t tS = tmem + Cfg::TMEM_S + (sc & 1) * 128 + lane_off;
                    tmem_ld_quad64(tS, s0);
                    tmem_ld_quad64(tS + 64, s1);
                    tc_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars.s_free[sc & 1]);
                    ++sc;
                    if (handed) {                               // the previous block's last stores are complete by now
                        if (lane == 0) { tma_store_wait_all(); st_release_cta(&stored[wq], ++nstored); }
                        handed = false;
                    }
                    if (j < It) hand_on(s0, own + (size_t)j * (S_BLOCK_BYTES / 4));
                } else {
                    // ---- a block computed by the CTA of tile j, read transposed
#pragma unroll
                    for (int half = 0; half < 2; ++half, ++mc) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&bars.m_full[mc % MST], (mc / MST) & 1, abortp));
                        if (!ok) break;
                        const float* src = reinterpret_cast<const float*>(sM + (mc % MST) * S_HALF_BYTES);
                        uint32_t (&s)[32] = half ? s1 : s0;
#pragma unroll
                        for (int g = 0; g < 4; ++g)             // keys 16 g .. 16 g + 15 of the half, row A / B, key parity
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const uint2 v = *reinterpret_cast<const uint2*>(src + ((e & 1) ? get_odd : get_even) + 2048 * g + 128 * (e >> 1));
                                s[8 * g + e] = v.x;
                                s[8 * g + 4 + e] = v.y;
                            }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars.m_empty[mc % MST]);
                    }
                    if (!ok) break;
                }
                // ---- keys beyond the sequence (ragged last block) carry no weight
                const int nvalid = n - j * TILE;
                if (nvalid < TILE) {
                    mask_quad64(s0, cq, nvalid - 1, nvalid - 1);
                    mask_quad64(s1, 64 + cq, nvalid - 1, nvalid - 1);
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
                // ---- P = exp2(S*sl2 - m) as bf16; its buffer is free behind the PV before the previous one
                const uint32_t tP = tmem + Cfg::TMEM_P + (blk & 1) * 64 + lane_off;
                float sumA = 0.f, sumB = 0.f;
                uint32_t pk[16];
                exp_quad64(s0, sl2, -mA, -mB, pk, sumA, sumB);
                if (j < It) {
                    hand_on(s1, own + (size_t)j * (S_BLOCK_BYTES / 4) + 1024);
                    handed = true;
                }
                if (blk >= 2) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars.o_done[blk & 1], ((blk >> 1) - 1) & 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
                }
                tmem_st_quad32(tP, pk);
                exp_quad64(s1, sl2, -mA, -mB, pk, sumA, sumB);
                tmem_st_quad32(tP + 32, pk);
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
                    for (int c = 0; c < D / 64; ++c) {
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
            const int bh = bh0 + hl, b = bh / H, h = bh - b * H;
            const float invA = 1.f / quad_sum(lA), invB = 1.f / quad_sum(lB);
#pragma unroll
            for (int u = 0; u < Cfg::SUB; ++u) {
                uint32_t v[32];
                tmem_ld_quad64(tO + 64 * u, v);
                tc_wait_ld();
                if (u == 0) {               // whatever used the buffer last must have been read
                    if (lane == 0) tma_store_wait_read();
                    __syncwarp();
                }
                uint8_t* sub = stage + u * (16 * 64 * 2);
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
                    tma_store_4d(&maps.o, sub, 64 * u, h, It * TILE + row0, b);
                    tma_store_commit();
                }
            }
            tc_fence_before();
        }
        if (wq == 0 && lane == 0) grid_launch_dependents();
        if (lane == 0) tma_store_wait_read();   // shared memory may be released; the writes complete on their own
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// The flags of `heads` heads and the work counter of a launch (the diagonal block whose place they take has room for 16384),
// cleared together with `before` bytes ahead of each of these places: for the first head, what lies ahead of the scratch;
// for the others the end of a diagonal block, which nothing uses.
cudaError_t sym_clear(float* S, int heads, int T, size_t before, cudaStream_t stream) {
    char* p = reinterpret_cast<char*>(S) - before;
    const size_t bytes = before + (size_t)(T + 1) * sizeof(int);
    return heads == 1 ? cudaMemsetAsync(p, 0, bytes, stream) : cudaMemset2DAsync(p, (size_t)sym_pairs(T) * S_BLOCK_BYTES, 0, bytes, heads, stream);
}

// Heads per group of the item list: the tiles of one head are started a group apart.  A tile needs its first handed-on block
// one step after its neighbour has computed it, so tiles that start together wait for one another; started 256 / T items
// apart (two steps, on 148 CTAs) they do not, and a head's scratch still lives briefly enough to stay in L2.  Measured for
// 64 / 128 / 256 / 512 / 1024 items (us; n = 256, 1024, 4096 at d_k = 128): 106 99 89 87 87, 279 270 249 252 258, 948 949 937
// 959 961.
constexpr int SYM_GROUP_ITEMS = 256;

// D: head size the kernel works with (64 or 128); d <= D: the tensors' head size (see the 4-D tensor maps).
// s_bytes: size of the score scratch, which sets the heads per pass; s_clear: the first pass finds its flags clear.
template <int D>
int launch_symmetric(const void* X, void* out, float* S, size_t s_bytes, bool s_clear, int B, int H, int n, int d, float scale, DeviceCounters* dc,
                     cudaStream_t stream) {
    using Cfg = SymCfg<D>;
    static DeviceSetup setup;
    const int sm_count = device_setup(&setup, [] {
        return cudaFuncSetAttribute(sym_attn_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, SymCfg<D>::SMEM);
    }, "cudaFuncSetAttribute(symmetric attention)");
    if (sm_count <= 0) return PSA_ERR_CUDA;
    const int T = row_tiles(n);
    const int hp = sym_heads_per_pass((size_t)B * H, n, s_bytes);
    SymMaps maps;
    if (!make_tensor_map_bf16_4d(&maps.x, X, B, n, H, d, 128) || !make_tensor_map_bf16_4d(&maps.o, out, B, n, H, d, 16))
        return PSA_ERR_CUDA;
    for (int bh0 = 0; bh0 < B * H; bh0 += hp) {
        const int heads = min(hp, B * H - bh0);
        if ((long long)heads * T > 0x7fffffffLL - 2 * sm_count) return PSA_ERR_SHAPE;      // (the work counter runs past the list)
        const int nitems = heads * T;
        cudaError_t e = bh0 == 0 && s_clear ? cudaSuccess : sym_clear(S, heads, T, 0, stream);
        if (e != cudaSuccess) { set_cuda_error(e, "symmetric scheme: clearing the flags"); return PSA_ERR_CUDA; }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(min(nitems, sm_count));
        cfg.blockDim = dim3(SYM_THREADS);
        cfg.dynamicSmemBytes = Cfg::SMEM;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, sym_attn_kernel<D>, maps, S, n, H, bh0, heads, min(heads, max(1, SYM_GROUP_ITEMS / T)), scale * LOG2E, dc);
        if (e != cudaSuccess) { set_cuda_error(e, "sym_attn_kernel launch"); return PSA_ERR_CUDA; }
    }
    return PSA_OK;
}

}  // namespace

cudaError_t bf16_symmetric_clear(float* S, size_t s_bytes, int B, int H, int n, size_t before, cudaStream_t stream) {
    return sym_clear(S, sym_heads_per_pass((size_t)B * H, n, s_bytes), row_tiles(n), before, stream);
}

int bf16_attention(const void* Q, const void* K, const void* V, void* out, float* S, size_t s_bytes, bool s_clear, int B, int H,
                   int n, int d, float scale, int scheme, DeviceCounters* dc, unsigned int* cursor, DeviceCounters* dc_next,
                   cudaStream_t stream) {
    if (scheme != PSA_SYMMETRIC && d > 128) return bf16_attention_wide(Q, K, V, out, B, H, n, d, scale, scheme, dc, cursor, dc_next, stream);
    if (scheme != PSA_SYMMETRIC) return bf16_attention_persist(Q, K, V, out, B, H, n, d, scale, scheme, dc, cursor, dc_next, stream);
    if (!S || s_bytes < (size_t)sym_pairs(row_tiles(n)) * S_BLOCK_BYTES) return PSA_ERR_WORKSPACE;       // (one head)
    if ((reinterpret_cast<uintptr_t>(S) & 15u) != 0) return PSA_ERR_ALIGN;
    if (d < 8 || d > 128 || d % 8) return PSA_ERR_UNSUPPORTED;
    if (d <= 64) return launch_symmetric<64>(Q, out, S, s_bytes, s_clear, B, H, n, d, scale, dc, stream);
    return launch_symmetric<128>(Q, out, S, s_bytes, s_clear, B, H, n, d, scale, dc, stream);
}

}  // namespace psa
