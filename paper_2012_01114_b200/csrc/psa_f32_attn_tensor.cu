// fp32 attention on the tensor cores (FULL and MASKED schemes, large calls), to the accuracy of the fp32 path.
//
// As in psa_f32_tensor.cu a number is the exact sum of three bf16 parts and a product the sum of six bf16 products (what is
// left out is below 2^-24 of it).  A block of 128 query rows by 64 keys takes
//     phase 1  S = Q K^T    the five small products of all columns first, the leading ones behind them into the same accumulator
//     phase 2  softmax      running maximum and sum in fp32, the weights split into parts in registers
//     phase 3  O = P V      in the same way; the accumulator holds one block and is added to the running output in fp32
//                           registers, so that no sum in the tensor core (which does not round to nearest) is longer than 8
// with Q and P read from tensor memory, K and V from shared memory.  K and V are split once per call by f32_split_kernel,
// Q once per row tile by the warps that need it.
//
// Skipping stays element-exact: under the masked scheme only blocks of keys before the row tile come here; the weights inside the
// tile (128 x 128, on the diagonal) are computed one by one by f32_diagonal_kernel (psa_f32.cu) ahead of this kernel, which
// continues from their maximum, sum and partial output.
//
// What the parts cannot carry: f32_split_kernel marks heads with an operand that is not finite, a number of Q or K beyond 2^50, a
// value (V) beyond 2^46 or a nonzero one below 2^-60; these are left to f32_flash_kernel altogether.  Weights are scaled by 2^64, so that
// every one that fp32 can hold has parts in the normal range.  With a maximum that may lag by FM_RAISE a weight is at most 2^64 e^4, and
// 1024 of them times 2^46 are below 2^126: the running output stays finite.  (Scores of 128 products of 2^100 are below 2^108.)
//
// What bounds it: per block of 64 keys 72 MMAs, 3072 cycles at d = 128 and 1536 at d = 64, beside about 1500 issue slots per scheduler of
// softmax and splitting; the masked scheme also its longest row tiles and the diagonal tiles ahead of them (30 of its 76 us at 16
// heads of n = 1024, d = 128).  Measured (us, CUDA cores before / whole call now): 16 heads of n = 1024, d = 128 FULL 308 / 54, MASKED
// 166 / 77; 48 of n = 512, d = 64, FULL 111 / 42.
// Error against 64 bits (relative, 2-norm; here / on CUDA cores; normal q, k, v): FULL 1.5e-7 .. 3.1e-7 / 2.1e-7 .. 4.8e-7, MASKED 1.4e-7 .. 2.4e-7 / 1.6e-7 ..
// 2.6e-7, nowhere more than 1 % larger.  Where all values have one sign the tensor core's rounding towards zero adds up, 1.0e-7 .. 1.2e-7, against 0.85e-7 .. 3.4e-7: more
// than on CUDA cores (by up to a quarter) only for FULL calls of few heads of up to 513 keys, whose sums those split in four.
//
// Roles (320 threads): warp 0 = TMA producer, warp 1 = MMA issuer, warps 2-9 = softmax, running output (a warp owns 16 rows, quad
// layout of sm100.cuh).  S of the next block is computed during the softmax of a block, its PV during the softmax of the next.
#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_softmax.cuh"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int FM_KEYS = 64;                              // keys of a block
constexpr int FM_WARPS = 8, FM_THREADS = 32 * (2 + FM_WARPS);
constexpr int FM_TMEM_Q = 0, FM_TMEM_S = 192, FM_TMEM_P = 256, FM_TMEM_O = 384;
constexpr float FM_UP = 1.8446744e19f;                   // 2^64
constexpr float FM_RAISE = 4.f;                          // the running maximum follows when a row's grew by more (natural units)
// Bits of 2^50, 2^46 and 2^-60: what the parts can carry, see above.
constexpr uint32_t FM_MOST = (127u + 50u) << 23, FM_VALUE_MOST = (127u + 46u) << 23, FM_VALUE_LEAST = (127u - 60u) << 23;

template <int D>
struct FMCfg {
    static constexpr int SUB = D / 64;
    static constexpr int PART_BYTES = FM_KEYS * D * 2;   // one part of a K or V tile
    static constexpr int STAGE_BYTES = 3 * PART_BYTES;
    static constexpr int STAGES = D == 128 ? 4 : 6;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
};
struct FMMaps {
    CUtensorMap k, v;      // parts of K and V as [3 * batch, n, heads, d] bf16, boxes of 64 rows x 64 columns
};

// The three parts of two numbers, packed (first: rounded, second: cut off, third: the rest).
__device__ __forceinline__ void split2(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    const uint32_t a0 = (__float_as_uint(a) + 0x8000u) & 0xffff0000u, b0 = (__float_as_uint(b) + 0x8000u) & 0xffff0000u;
    const float ra = a - __uint_as_float(a0), rb = b - __uint_as_float(b0);
    const uint32_t a1 = __float_as_uint(ra) & 0xffff0000u, b1 = __float_as_uint(rb) & 0xffff0000u;
    p0 = __byte_perm(a0, b0, 0x7632);
    p1 = __byte_perm(a1, b1, 0x7632);
    p2 = __byte_perm(__float_as_uint(ra - __uint_as_float(a1)), __float_as_uint(rb - __uint_as_float(b1)), 0x7632);
}

// blockIdx.y: 0 K, 1 V, 2 Q (looked at only).  `count4`: groups of four numbers of a tensor.
__global__ void __launch_bounds__(256)
f32_split_kernel(const float4* __restrict__ Q, const float4* __restrict__ K, const float4* __restrict__ V, uint2* __restrict__ parts, uint32_t count4,
                 int d, int H, int n, int* __restrict__ bad, int mark) {
    const int which = blockIdx.y;
    const float4* src = which == 0 ? K : (which == 1 ? V : Q);
    uint2* dst = parts + (size_t)which * 3 * count4;
    grid_dependency_wait();
    for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < count4; i += gridDim.x * 256u) {
        const float4 x = __ldg(src + i);
        const uint32_t most = max(max(__float_as_uint(x.x) & 0x7fffffffu, __float_as_uint(x.y) & 0x7fffffffu),
                                  max(__float_as_uint(x.z) & 0x7fffffffu, __float_as_uint(x.w) & 0x7fffffffu));
        // (twice the bits less one: zero becomes the largest)
        const uint32_t least = min(min(2u * __float_as_uint(x.x) - 1u, 2u * __float_as_uint(x.y) - 1u), min(2u * __float_as_uint(x.z) - 1u, 2u * __float_as_uint(x.w) - 1u));
        if (most > (which == 1 ? FM_VALUE_MOST : FM_MOST) || (which == 1 && least < 2u * FM_VALUE_LEAST - 1u)) {
            const uint32_t row = i / (uint32_t)(d >> 2);
            bad[(row / ((uint32_t)n * H)) * H + row % (uint32_t)H] = mark;
        }
        if (which == 2) continue;
        uint2 p[3];
        split2(x.x, x.y, p[0].x, p[1].x, p[2].x);
        split2(x.z, x.w, p[0].y, p[1].y, p[2].y);
#pragma unroll
        for (int k = 0; k < 3; ++k) dst[(size_t)k * count4 + i] = p[k];
    }
}

template <int D>
__global__ void __launch_bounds__(FM_THREADS, 1)
f32_attn_tensor_kernel(const __grid_constant__ FMMaps maps, const float* __restrict__ Q, float* __restrict__ out, const float* __restrict__ ml,
                       const int* __restrict__ bad, int mark, int B, int H, int n, int d, int masked, int nitems, float scale, DeviceCounters* dc) {
    using Cfg = FMCfg<D>;
    constexpr int ST = Cfg::STAGES;
    extern __shared__ uint8_t fm_smem_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(fm_smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[ST], empty[ST], q_ready, s_full, s_free, p_ready, o_done;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int T = row_tiles(n), BH = B * H;
    // FULL: head by head.  MASKED: the longest row tiles of all heads first; the first tile of a head has nothing to do here.
    auto item_work = [&](int idx, int& bh, int& It, int& nblk) {
        if (masked) {
            const int r = idx / BH;
            It = T - 1 - r;
            bh = idx - r * BH;
            nblk = It * (TILE / FM_KEYS);
        } else {
            bh = idx / T;
            It = idx - bh * T;
            nblk = (n + FM_KEYS - 1) / FM_KEYS;
        }
    };

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < ST; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(&q_ready, FM_WARPS);
        mbar_init(&s_full, 1);
        mbar_init(&s_free, FM_WARPS);
        mbar_init(&p_ready, FM_WARPS);
        mbar_init(&o_done, 1);
        fence_mbar_init();
    }
    if (warp == 1) { tmem_alloc(&tmem_base_s, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;
    grid_dependency_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------------ TMA producer: K_0, K_1, V_0, K_2, V_1, ...
            uint32_t rc = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < nitems && ok; idx += gridDim.x) {
                int bh, It, nblk;
                item_work(idx, bh, It, nblk);
                if (bad[bh] == mark) continue;
                const int b = bh / H, h = bh - b * H;
                auto load = [&](const CUtensorMap* map, int j) {
                    const int s = rc % ST;
                    if (rc >= (uint32_t)ST) ok = mbar_wait(&empty[s], ((rc / ST) - 1) & 1, abortp);
                    if (!ok) return;
                    mbar_arrive_expect_tx(&full[s], Cfg::STAGE_BYTES);
                    for (int p = 0; p < 3; ++p)
                        for (int u = 0; u < Cfg::SUB; ++u)
                            tma_load_4d(ring + s * Cfg::STAGE_BYTES + p * Cfg::PART_BYTES + u * 8192, map, &full[s], 64 * u, h, j * FM_KEYS, p * B + b);
                    ++rc;
                };
                load(&maps.k, 0);
                for (int j = 0; j < nblk && ok; ++j) {
                    if (j + 1 < nblk) load(&maps.k, j + 1);
                    if (ok) load(&maps.v, j);
                }
            }
            if (*abortp)      // let copies already issued land before shared memory is released
                for (uint32_t c = rc > (uint32_t)ST ? rc - ST : 0; c < rc; ++c) mbar_wait_drain(&full[c % ST], (c / ST) & 1);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // ------------------------------------------------------------ MMA issuer
            const uint32_t idescS = umma_idesc_bf16(128, FM_KEYS, UMMA_K_MAJOR, UMMA_K_MAJOR);
            const uint32_t idescO = umma_idesc_bf16(128, D, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t k_lo = umma_desc_lo_kmajor(smem_u32(ring)), v_lo = umma_desc_lo_mnmajor(smem_u32(ring), 8192);
            constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};      // the leading product last
            uint32_t rc = 0, blk = 0, items = 0;
            bool ok = true;
            auto issue_S = [&](bool wait_free) -> bool {
                const uint32_t s = rc % ST;
                if (!mbar_wait(&full[s], (rc / ST) & 1, abortp)) return false;
                if (wait_free && !mbar_wait(&s_free, (blk - 1) & 1, abortp)) return false;
                tc_fence_after();
                const uint32_t k = k_lo + s * (Cfg::STAGE_BYTES >> 4);
#pragma unroll
                for (int t = 0; t < 6; ++t)
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        umma_ts(tmem + FM_TMEM_S, tmem + FM_TMEM_Q + PA[t] * (D / 2) + kk * 8,
                                umma_desc_join(k + ((PB[t] * Cfg::PART_BYTES + (kk >> 2) * 8192 + (kk & 3) * 32) >> 4), UMMA_DESC_HI_SW128), idescS,
                                t != 0 || kk != 0);
                umma_commit(&s_full);
                umma_commit(&empty[s]);
                ++rc;
                ++blk;                 // S issued so far
                return true;
            };
            unsigned long long macs = 0;
            for (int idx = blockIdx.x; idx < nitems && ok; idx += gridDim.x) {
                int bh, It, nblk;
                item_work(idx, bh, It, nblk);
                if (bad[bh] == mark) continue;
                ok = mbar_wait(&q_ready, items & 1, abortp) && issue_S(blk > 0);
                ++items;
                for (int j = 0; j < nblk && ok; ++j) {
                    const uint32_t pv = blk - 1;                       // number of block j
                    if (j + 1 < nblk) ok = issue_S(true);
                    const uint32_t s = rc % ST;
                    if (ok) ok = mbar_wait(&full[s], (rc / ST) & 1, abortp) && mbar_wait(&p_ready, pv & 1, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t v = v_lo + s * (Cfg::STAGE_BYTES >> 4);
#pragma unroll
                    for (int t = 0; t < 6; ++t)
#pragma unroll
                        for (int kk = 0; kk < FM_KEYS / 16; ++kk)
                            umma_ts(tmem + FM_TMEM_O, tmem + FM_TMEM_P + PA[t] * (FM_KEYS / 2) + kk * 8,
                                    umma_desc_join(v + ((PB[t] * Cfg::PART_BYTES + kk * 2048) >> 4), UMMA_DESC_HI_SW128), idescO, t != 0 || kk != 0);
                    umma_commit(&o_done);
                    umma_commit(&empty[s]);
                    ++rc;
                    macs += (unsigned long long)min(TILE, n - It * TILE) * min(FM_KEYS, n - j * FM_KEYS);
                }
            }
            if (macs) {
                atomicAdd(&dc->qk_macs, macs * d);
                atomicAdd(&dc->pv_macs, macs * d);
                atomicAdd(&dc->exps, macs);
            }
        }
    } else {
        // ------------------------------------------------------------ Q parts, softmax, running output
        const int wq = warp - 2, q = warp & 3;
        const int row0 = q * 32 + (wq >> 2) * 16;               // first of the warp's 16 rows inside the tile
        const int rA = row0 + (lane >> 2);                      // this thread's rows: rA and rA + 8
        const int cq = 2 * (lane & 3);
        const uint32_t lanes = tmem + (static_cast<uint32_t>(row0) << 16);
        uint32_t blk = 0;                                       // blocks so far, all items
        bool ok = true;
        for (int idx = blockIdx.x; idx < nitems && ok; idx += gridDim.x) {
            int bh, It, nblk;
            item_work(idx, bh, It, nblk);
            if (bad[bh] == mark) continue;
            const int b = bh / H, h = bh - b * H, gA = It * TILE + rA, gB = gA + 8;
            const size_t at = (((size_t)b * n + gA) * H + h) * d, down = (size_t)8 * H * d;
            // ---- the row tile's Q, split into tensor memory (every S of the item before has been waited for)
#pragma unroll
            for (int c = 0; c < Cfg::SUB; ++c) {
                uint32_t p0[16], p1[16], p2[16];
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const int col = 64 * c + 8 * g + cq;
                    const float2 zero = make_float2(0.f, 0.f);
                    const float2 a = gA < n && col < d ? __ldg(reinterpret_cast<const float2*>(Q + at + col)) : zero;
                    const float2 e = gB < n && col < d ? __ldg(reinterpret_cast<const float2*>(Q + at + down + col)) : zero;
                    split2(a.x, a.y, p0[2 * g], p1[2 * g], p2[2 * g]);
                    split2(e.x, e.y, p0[2 * g + 1], p1[2 * g + 1], p2[2 * g + 1]);
                }
                tmem_st_quad32(lanes + FM_TMEM_Q + 32 * c, p0);
                tmem_st_quad32(lanes + FM_TMEM_Q + D / 2 + 32 * c, p1);
                tmem_st_quad32(lanes + FM_TMEM_Q + D + 32 * c, p2);
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&q_ready);
            // ---- the running output: columns 64 c + 8 g + cq, + 1 of rows A and B
            float mA = -INFINITY, mB = -INFINITY, lA = 0.f, lB = 0.f;
            float acc[Cfg::SUB][32];
#pragma unroll
            for (int c = 0; c < Cfg::SUB; ++c)
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[c][e] = 0.f;
            if (masked) {            // continued from the weights inside the tile (a whole tile but for the sequence's end)
                const float* mp = ml + (size_t)bh * n + gA;
                const float* lp = mp + (size_t)BH * n;
                if (gA < n) { mA = mp[0]; lA = (lane & 3) == 0 ? lp[0] * FM_UP : 0.f; }
                if (gB < n) { mB = mp[8]; lB = (lane & 3) == 0 ? lp[8] * FM_UP : 0.f; }
#pragma unroll
                for (int c = 0; c < Cfg::SUB; ++c)
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        const int col = 64 * c + 8 * g + cq;
                        if (gA < n && col < d) {
                            const float2 y = *reinterpret_cast<const float2*>(out + at + col);
                            acc[c][4 * g] = y.x * FM_UP; acc[c][4 * g + 1] = y.y * FM_UP;
                        }
                        if (gB < n && col < d) {
                            const float2 y = *reinterpret_cast<const float2*>(out + at + down + col);
                            acc[c][4 * g + 2] = y.x * FM_UP; acc[c][4 * g + 3] = y.y * FM_UP;
                        }
                    }
            }
            auto drain = [&](uint32_t pv) -> bool {             // adds the output of block pv
                if (!__all_sync(0xffffffffu, mbar_wait(&o_done, pv & 1, abortp))) return false;
                tc_fence_after();
#pragma unroll
                for (int c = 0; c < Cfg::SUB; ++c) {
                    uint32_t v[32];
                    tmem_ld_quad64(lanes + FM_TMEM_O + 64 * c, v);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) acc[c][e] += __uint_as_float(v[e]);
                }
                return true;
            };
            for (int j = 0; j < nblk; ++j, ++blk) {
                ok = __all_sync(0xffffffffu, mbar_wait(&s_full, blk & 1, abortp));
                if (!ok) break;
                uint32_t s[32];
                tc_fence_after();
                tmem_ld_quad64(lanes + FM_TMEM_S, s);
                tc_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_free);
#pragma unroll
                for (int e = 0; e < 32; ++e) s[e] = __float_as_uint(__uint_as_float(s[e]) * scale);
                const int last = n - 1 - j * FM_KEYS;           // keys beyond the sequence carry no weight
                if (last < FM_KEYS - 1) mask_quad64(s, cq, last, last);
                float bA = -INFINITY, bB = -INFINITY;
                max_quad64(s, bA, bB);
                bA = quad_max(bA);
                bB = quad_max(bB);
                float fA = 1.f, fB = 1.f;                       // what the running output is multiplied by
                if (bA > mA + FM_RAISE) { fA = expf(mA - bA); mA = bA; }
                if (bB > mB + FM_RAISE) { fB = expf(mB - bB); mB = bB; }
                float sumA = 0.f, sumB = 0.f;
                uint32_t p0[16], p1[16], p2[16];
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const float w0 = expf(__uint_as_float(s[4 * g]) - mA) * FM_UP, w1 = expf(__uint_as_float(s[4 * g + 1]) - mA) * FM_UP;
                    const float w2 = expf(__uint_as_float(s[4 * g + 2]) - mB) * FM_UP, w3 = expf(__uint_as_float(s[4 * g + 3]) - mB) * FM_UP;
                    sumA += w0 + w1;
                    sumB += w2 + w3;
                    split2(w0, w1, p0[2 * g], p1[2 * g], p2[2 * g]);
                    split2(w2, w3, p0[2 * g + 1], p1[2 * g + 1], p2[2 * g + 1]);
                }
                // P and O are in use by the PV of the block before until its commit
                if (j > 0 && !drain(blk - 1)) { ok = false; break; }
                tc_fence_after();
                tmem_st_quad32(lanes + FM_TMEM_P, p0);
                tmem_st_quad32(lanes + FM_TMEM_P + 32, p1);
                tmem_st_quad32(lanes + FM_TMEM_P + 64, p2);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&p_ready);
                lA = fmaf(lA, fA, sumA);
                lB = fmaf(lB, fB, sumB);
                if (__any_sync(0xffffffffu, fA != 1.f || fB != 1.f)) {
#pragma unroll
                    for (int c = 0; c < Cfg::SUB; ++c)
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            acc[c][4 * g] *= fA; acc[c][4 * g + 1] *= fA;
                            acc[c][4 * g + 2] *= fB; acc[c][4 * g + 3] *= fB;
                        }
                }
            }
            if (!ok) break;
            ok = drain(blk - 1);
            if (!ok) break;
            tc_fence_before();
            const float invA = 1.f / quad_sum(lA), invB = 1.f / quad_sum(lB);
#pragma unroll
            for (int c = 0; c < Cfg::SUB; ++c)
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const int col = 64 * c + 8 * g + cq;
                    if (gA < n && col < d) *reinterpret_cast<float2*>(out + at + col) = make_float2(acc[c][4 * g] * invA, acc[c][4 * g + 1] * invA);
                    if (gB < n && col < d) *reinterpret_cast<float2*>(out + at + down + col) = make_float2(acc[c][4 * g + 2] * invB, acc[c][4 * g + 3] * invB);
                }
        }
        if (wq == 0 && lane == 0) grid_launch_dependents();
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == 1) tmem_dealloc(tmem, 512);
}

template <int D>
cudaError_t launch_main(const float* Q, float* out, const F32Scratch& fs, int B, int H, int n, int d, float scale, int masked, DeviceCounters* dc,
                        cudaStream_t stream) {
    using Cfg = FMCfg<D>;
    static DeviceSetup setup;
    const int sms = device_setup(&setup, [] {
        return cudaFuncSetAttribute(f32_attn_tensor_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, FMCfg<D>::SMEM);
    }, "fp32 tensor attention set-up");
    if (sms <= 0) return cudaErrorUnknown;
    const size_t part = (size_t)B * n * H * d * 2;
    FMMaps maps;
    if (!make_tensor_map_bf16_4d(&maps.k, fs.parts, 3 * (uint64_t)B, n, H, d, FM_KEYS) ||
        !make_tensor_map_bf16_4d(&maps.v, static_cast<char*>(fs.parts) + 3 * part, 3 * (uint64_t)B, n, H, d, FM_KEYS))
        return cudaErrorInvalidValue;
    const int T = row_tiles(n), nitems = B * H * (masked ? T - 1 : T);
    if (nitems == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nitems < sms ? nitems : sms);
    cfg.blockDim = dim3(FM_THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f32_attn_tensor_kernel<D>, maps, Q, out, static_cast<const float*>(fs.ml), static_cast<const int*>(fs.bad), fs.mark, B, H, n, d,
                              masked, nitems, scale, dc);
}

}  // namespace

cudaError_t f32_attention_split(const float* Q, const float* K, const float* V, const F32Scratch& fs, int B, int H, int n, int d, cudaStream_t stream) {
    const uint32_t count4 = (uint32_t)((size_t)B * n * H * d / 4);
    const uint32_t blocks = (count4 + 1023) / 1024;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks < 1024 ? blocks : 1024, 3);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f32_split_kernel, reinterpret_cast<const float4*>(Q), reinterpret_cast<const float4*>(K), reinterpret_cast<const float4*>(V),
                              static_cast<uint2*>(fs.parts), count4, d, H, n, fs.bad, fs.mark);
}
cudaError_t f32_attention_tensor(const float* Q, float* out, const F32Scratch& fs, int B, int H, int n, int d, float scale, int masked, DeviceCounters* dc,
                                 cudaStream_t stream) {
    return d <= 64 ? launch_main<64>(Q, out, fs, B, H, n, d, scale, masked, dc, stream) : launch_main<128>(Q, out, fs, B, H, n, d, scale, masked, dc, stream);
}

}  // namespace psa
