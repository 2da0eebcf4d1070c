// Projection of the fp32 path on the tensor cores: C_w[M, N] = X[M, K] * W_w[K, N] (+ R[M, N]), fp32 in and out, to the
// accuracy of an fp32 sum.
//
// An fp32 number is the sum of three bf16 numbers (8 + 8 + 8 significant bits; the two remainders are exact), so a product is
// the sum of nine bf16 products, of which the six largest are formed; the other three are below 2^-24 of it.  The tensor
// core adds bf16 products into fp32 accumulators, but it was not made to keep the last bits of long sums, so
//   * the leading products (first part times first part) of 128 consecutive k go to an accumulator of their own, which is
//     read and added, rounded as usual, to the running sum in registers: 8 additions in the tensor core, not K / 16;
//   * the five smaller products go to a second accumulator, 2^-8 of the first in size, read once per tile.
// Measured against 64 bits (relative, 2-norm; normal inputs): K = 320 / 768 / 2048 1.2e-7 / 1.3e-7 / 1.5e-7, where the plain
// chain of fmaf has 3.2e-7 / 5.0e-7 / 8.1e-7; positive inputs, K = 768, 1.4e-7 (of which 1.3e-7 is the accumulators' rounding
// towards zero) against 4.3e-7.
//
// f32_project_tensor_kernel: a CTA takes tiles of 128 x 128.  Warps 0-15 read X and W (two steps of 32 k ahead, in registers), split them into parts
// and write these as operand tiles in the 128-byte swizzle (X K-major, W MN-major) into a ring of four steps; warp 16
// issues 12 MMAs of 128 x 128 x 16 per step; warps 0-15 also drain the accumulators, 32 rows by 32 columns each.
//
// What bounds it: 12 MMAs per step at 64 cycles (N = 128) are 768 cycles for 32 k; splitting a step takes about 600 issue
// slots per scheduler beside them, and its stores share the shared-memory port with the MMAs' operands (at the 96 registers
// that 17 warps leave, 92 bytes are spilled, most of them around the call of ft_form_again).  Measured 2300 cycles per step;
// 2048 x 768 x 3 x 768 171 us on CUDA cores (128 x 128 tiles), 70 us here.
//
// What the parts cannot carry is formed again by the plain chain of fmaf, per output (ft_form_again):
//   * an output that is not finite (an input is infinite or NaN or rounds to infinity, or a sum overflows);
//   * an output of a tile with a nonzero operand below 2^-60, if it is small enough to have lost something: an operand below
//     2^-100 has parts below the normal range of bf16 and loses up to 2^-125, and products below 2^-120 lose up to 2^-149 in
//     each addition.  With the largest magnitudes of the output's row and column that bounds its error, K times over; it is
//     formed again where that could be more than half a unit.
// Such tiles are marked on the way and looked at when the CTA's other work is done, so that the main loop keeps its registers.
// What it cost, in a layer of 4 x 512 vectors, d_model = 768, 12 heads, of whose 176 us the projection took 60: one 1e-35 in
// every vector, so that every tile is looked at, 208 us; nothing but numbers around 1e-33, so that every output is formed
// again, 439; nothing but NaN 416 (as a loop of one thread per 32 outputs in global memory it was 3300 in all three).
#include "psa_internal.h"
#include "psa_tma.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int FT_M = 128, FT_N = 128, FT_K = 32;         // tile, depth of a step
constexpr int FT_WORKERS = 16, FT_THREADS = 32 * (FT_WORKERS + 1);
constexpr int FT_PLANE_BYTES = 128 * 64 * 2;             // one part of an operand over two steps: 16 KB
constexpr int FT_BUF_BYTES = 6 * FT_PLANE_BYTES;         // X parts 0-2, W parts 0-2 of two steps
constexpr int FT_SLOTS = 4;                              // steps in the ring (two buffers of two)
constexpr int FT_CHUNK = 4;                              // steps whose leading products share an accumulator pass
constexpr int FT_SMEM = FT_SLOTS / 2 * FT_BUF_BYTES + 1024;
constexpr int FT_TMEM_MAIN = 0, FT_TMEM_CROSS = 256;     // leading products (two accumulators), smaller products
constexpr uint32_t FT_SMALL = 2u * (67u << 23), FT_TINY = 2u * (27u << 23);      // twice the bits of 2^-60, 2^-100
constexpr int FT_MARKS = 1024;                           // marks of a CTA's tiles
constexpr int FT_PITCH = 36;                             // floats per row of a warp's 32 x 32 output staging

__device__ __forceinline__ uint32_t ft_pack(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }    // upper halves

// The three parts of four numbers, packed as bf16 and written to the same place of three planes: the first rounded to its 8
// bits, the second cut off, the third what is left (at most 8 bits).
// `least` becomes the smallest of twice the bits of the nonzero magnitudes, less one.
__device__ __forceinline__ void ft_split_store(uint8_t* dst, const float4& v, uint32_t& least) {
    const float x[4] = {v.x, v.y, v.z, v.w};
    uint32_t p[3][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        least = min(least, 2u * __float_as_uint(x[e]) - 1u);
        p[0][e] = (__float_as_uint(x[e]) + 0x8000u) & 0xffff0000u;
        const float r1 = x[e] - __uint_as_float(p[0][e]);
        p[1][e] = __float_as_uint(r1) & 0xffff0000u;
        p[2][e] = __float_as_uint(r1 - __uint_as_float(p[1][e]));
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        *reinterpret_cast<uint2*>(dst + k * FT_PLANE_BYTES) = make_uint2(ft_pack(p[k][0], p[k][1]), ft_pack(p[k][2], p[k][3]));
}

// Shared memory of ft_form_again, over the ring: 32 k of the operands as they are (X rows padded by 16 bytes), and twice the
// bits of the smallest nonzero magnitude (less one) and of the largest, per row of X and column of W.
struct FtAgain {
    float x[FT_M * (FT_K + 4)], w[FT_K * FT_N];
    uint32_t row_least[FT_M], row_most[FT_M], col_least[FT_N], col_most[FT_N];
};
static_assert(sizeof(FtAgain) <= FT_BUF_BYTES, "does not fit the ring");

// Replaces those outputs of a finished tile of 128 rows and 128 columns that the parts cannot carry, by the plain chain: called by
// WORKERS warps (16 or 8).  A thread has the eight rows row0 + 4 i and the four columns from col0 on (and, of eight warps, from col0 +
// 64 on: with four columns the loads from shared memory were the limit, 750 us for 4096 x 768 x 3 x 768).  Without a residual the outputs say whether there is
// anything to replace; with one the tile is computed again in any case.
template <int WORKERS>
__device__ __noinline__ void ft_form_again(const float* X, const float* W, float* O, const float* R, int m_first, int n_first, int M, int K,
                                           int N, FtAgain* sm) {
    constexpr int COLS = FT_N, CG = 16 / WORKERS, XU = FT_M * FT_K / (128 * WORKERS), WU = FT_K * COLS / (128 * WORKERS);     // 16-byte loads per thread
    const int tid = threadIdx.x % (32 * WORKERS), warp = tid >> 5, lane = tid & 31;
    const int row0 = 32 * (warp & 3) + (lane >> 3), col0 = 32 * (warp >> 2) + 4 * (lane & 7);
    named_bar_sync(1, 32 * WORKERS);       // (the tile before is done with the shared memory)
    if (tid < FT_M) { sm->row_least[tid] = sm->col_least[tid] = 0xffffffffu; sm->row_most[tid] = sm->col_most[tid] = 0; }
    named_bar_sync(1, 32 * WORKERS);
    for (int r = warp; r < FT_M && m_first + r < M; r += WORKERS) {
        uint32_t least = 0xffffffffu, most = 0;
#pragma unroll 4
        for (int k = 4 * lane; k < K; k += 128) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(X + (size_t)(m_first + r) * K + k));
            const uint32_t t[4] = {2u * __float_as_uint(v.x), 2u * __float_as_uint(v.y), 2u * __float_as_uint(v.z), 2u * __float_as_uint(v.w)};
#pragma unroll
            for (int e = 0; e < 4; ++e) { least = min(least, t[e] - 1u); most = max(most, t[e]); }
        }
        least = __reduce_min_sync(0xffffffffu, least);
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0) { sm->row_least[r] = least; sm->row_most[r] = most; }
    }
    if (4 * lane < COLS && n_first + 4 * lane < N) {
        uint32_t least[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu}, most[4] = {0, 0, 0, 0};
#pragma unroll 8
        for (int k = warp; k < K; k += WORKERS) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(W + (size_t)k * N + n_first + 4 * lane));
            const uint32_t t[4] = {2u * __float_as_uint(v.x), 2u * __float_as_uint(v.y), 2u * __float_as_uint(v.z), 2u * __float_as_uint(v.w)};
#pragma unroll
            for (int e = 0; e < 4; ++e) { least[e] = min(least[e], t[e] - 1u); most[e] = max(most[e], t[e]); }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) { atomicMin(&sm->col_least[4 * lane + e], least[e]); atomicMax(&sm->col_most[4 * lane + e], most[e]); }
    }
    named_bar_sync(1, 32 * WORKERS);
    auto inside = [&](int cg) { return n_first + col0 + 64 * cg < N; };      // (N is a multiple of 4)
    float* out = O + (size_t)(m_first + row0) * N + n_first + col0;
    auto lost = [&](float v, int r, int c) {                // whether value v at (r, c) may have lost something
        if (!(fabsf(v) < INFINITY)) return true;
        if (sm->row_most[r] == 0 || sm->col_most[c] == 0) return false;       // a row or column of zeros gives exact zeros
        float limit = 7.5231638e-37f;                                         // 2^-120
        if (sm->row_least[r] < FT_TINY) limit += 7.8886091e-31f * __uint_as_float(sm->col_most[c] >> 1);       // 2^-100
        if (sm->col_least[c] < FT_TINY) limit += 7.8886091e-31f * __uint_as_float(sm->row_most[r] >> 1);
        return !(fabsf(v) >= limit * (float)K);
    };
    if (!R) {
        bool any = false;
        for (int i = 0; i < 8 * CG; ++i) {
            const int cg = i >> 3, rr = row0 + 4 * (i & 7), c = col0 + 64 * cg;
            if (!inside(cg) || m_first + rr >= M) continue;
            const float4 o = *reinterpret_cast<const float4*>(out + (size_t)(4 * (i & 7)) * N + 64 * cg);
            any = any || lost(o.x, rr, c) || lost(o.y, rr, c + 1) || lost(o.z, rr, c + 2) || lost(o.w, rr, c + 3);
        }
        if (named_bar_all(!any, 1, 32 * WORKERS)) return;
    }
    float acc[CG][8][4] = {};
    float4 xv[XU], wv[WU];                                  // the operands of the next 32 k
    auto fetch = [&](int k0) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < XU; ++u) {
            const int t = tid + 32 * WORKERS * u, m = m_first + (t >> 3), kx = k0 + 4 * (t & 7);
            xv[u] = m < M && kx < K ? __ldg(reinterpret_cast<const float4*>(X + (size_t)m * K + kx)) : zero;
        }
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int t = tid + 32 * WORKERS * u, kw = k0 + t / (COLS / 4), n = n_first + 4 * (t % (COLS / 4));
            wv[u] = kw < K && n < N ? __ldg(reinterpret_cast<const float4*>(W + (size_t)kw * N + n)) : zero;
        }
    };
    constexpr bool AHEAD = WORKERS <= 8;                    // (sixteen warps have no registers for it)
    if (AHEAD) fetch(0);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += FT_K) {
        if (!AHEAD) fetch(k0);
        named_bar_sync(1, 32 * WORKERS);
#pragma unroll
        for (int u = 0; u < XU; ++u) {
            const int t = tid + 32 * WORKERS * u;
            *reinterpret_cast<float4*>(sm->x + (t >> 3) * (FT_K + 4) + 4 * (t & 7)) = xv[u];
        }
#pragma unroll
        for (int u = 0; u < WU; ++u) *reinterpret_cast<float4*>(sm->w + 4 * (tid + 32 * WORKERS * u)) = wv[u];
        named_bar_sync(1, 32 * WORKERS);
        if (AHEAD) fetch(k0 + FT_K);
        const int kn = min(FT_K, K - k0);     // (a multiple of 4)
#pragma unroll 1
        for (int k = 0; k < kn; k += 4) {
            float4 w[CG][4];
#pragma unroll
            for (int cg = 0; cg < CG; ++cg)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) w[cg][kk] = *reinterpret_cast<const float4*>(sm->w + (k + kk) * COLS + col0 + 64 * cg);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(sm->x + (row0 + 4 * i) * (FT_K + 4) + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float f = kk == 0 ? x.x : kk == 1 ? x.y : kk == 2 ? x.z : x.w;
#pragma unroll
                    for (int cg = 0; cg < CG; ++cg) {
                        acc[cg][i][0] = fmaf(f, w[cg][kk].x, acc[cg][i][0]); acc[cg][i][1] = fmaf(f, w[cg][kk].y, acc[cg][i][1]);
                        acc[cg][i][2] = fmaf(f, w[cg][kk].z, acc[cg][i][2]); acc[cg][i][3] = fmaf(f, w[cg][kk].w, acc[cg][i][3]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int cg = 0; cg < CG; ++cg)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = row0 + 4 * i, c = col0 + 64 * cg;
            if (!inside(cg) || m_first + r >= M) continue;
            const size_t at = (size_t)(4 * i) * N + 64 * cg;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float o = out[at + e], v = acc[cg][i][e];
                if (!(fabsf(o) < INFINITY) || lost(R ? v : o, r, c + e)) out[at + e] = R ? v + R[(size_t)(m_first + r) * N + n_first + c + e] : v;
            }
        }
}

__global__ void __launch_bounds__(FT_THREADS, 1)
f32_project_tensor_kernel(const float* __restrict__ X, const float* W0, const float* W1, const float* W2, float* O0, float* O1,
                          float* O2, int M, int K, int N, int nW, const float* __restrict__ R, DeviceCounters* dc) {
    extern __shared__ uint8_t ft_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ft_smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full_bar[FT_SLOTS], empty_bar[FT_SLOTS], main_full[2], main_empty[2], cross_full, cross_empty;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;
    __shared__ uint32_t marks[FT_MARKS / 32];      // tiles of this CTA to look at again: see mark_of

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = (M + FT_M - 1) / FT_M, nt = (N + FT_N - 1) / FT_N, ntiles = mt * nt * nW;
    const int nsteps = 2 * ((K + 2 * FT_K - 1) / (2 * FT_K));         // an even number: the loads are two steps ahead

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < FT_SLOTS; ++s) { mbar_init(&full_bar[s], FT_WORKERS); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&main_full[b], 1); mbar_init(&main_empty[b], FT_WORKERS); }
        mbar_init(&cross_full, 1);
        mbar_init(&cross_empty, FT_WORKERS);
        fence_mbar_init();
    }
    for (int i = threadIdx.x; i < FT_MARKS / 32; i += FT_THREADS) marks[i] = 0;
    if (warp == FT_WORKERS) { tmem_alloc(&tmem_base_s, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;

    if (warp == FT_WORKERS) {
        if (lane == 0) {
            // ---- MMA issuer
            const uint32_t idesc = umma_idesc_bf16(FT_M, FT_N, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t a_lo0 = umma_desc_lo_kmajor(smem_u32(smem));
            const uint32_t b_lo0 = umma_desc_lo_mnmajor(smem_u32(smem + 3 * FT_PLANE_BYTES), FT_PLANE_BYTES / 2);
            unsigned long long macs = 0;
            uint32_t g = 0, gc = 0, i = 0;               // steps, chunks and tiles so far
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
                if (i > 0) ok = mbar_wait(&cross_empty, (i - 1) & 1, abortp);
                for (int s = 0; s < nsteps && ok; ++s, ++g) {
                    const int slot = g % FT_SLOTS;
                    const bool first = s % FT_CHUNK == 0;
                    if (first && gc >= 2) ok = mbar_wait(&main_empty[gc & 1], ((gc >> 1) - 1) & 1, abortp);
                    if (ok) ok = mbar_wait(&full_bar[slot], (g / FT_SLOTS) & 1, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = a_lo0 + (slot >> 1) * (FT_BUF_BYTES >> 4) + (slot & 1) * (64 >> 4);
                    const uint32_t b = b_lo0 + (slot >> 1) * (FT_BUF_BYTES >> 4) + (slot & 1) * (4096 >> 4);
                    auto mma = [&](uint32_t d, int pa, int pb, int k, uint32_t accumulate) {
                        umma_ss(d, umma_desc_join(a + pa * (FT_PLANE_BYTES >> 4) + k * (32 >> 4), UMMA_DESC_HI_SW128),
                                umma_desc_join(b + pb * (FT_PLANE_BYTES >> 4) + k * (2048 >> 4), UMMA_DESC_HI_SW128), idesc, accumulate);
                    };
                    const uint32_t dm = tmem + FT_TMEM_MAIN + (gc & 1) * FT_N, dx = tmem + FT_TMEM_CROSS;
                    mma(dm, 0, 0, 0, !first);
                    mma(dx, 0, 1, 0, s != 0);
                    mma(dx, 1, 0, 0, 1);
                    mma(dx, 1, 1, 0, 1);
                    mma(dx, 0, 2, 0, 1);
                    mma(dx, 2, 0, 0, 1);
                    mma(dm, 0, 0, 1, 1);
                    mma(dx, 0, 1, 1, 1);
                    mma(dx, 1, 0, 1, 1);
                    mma(dx, 1, 1, 1, 1);
                    mma(dx, 0, 2, 1, 1);
                    mma(dx, 2, 0, 1, 1);
                    umma_commit(&empty_bar[slot]);
                    if (s % FT_CHUNK == FT_CHUNK - 1 || s == nsteps - 1) { umma_commit(&main_full[gc & 1]); ++gc; }
                }
                if (!ok) break;
                umma_commit(&cross_full);
                const int r = t / nt;
                macs += (unsigned long long)min(FT_M, M - (r % mt) * FT_M) * min(FT_N, N - (t % nt) * FT_N) * K;
            }
            if (macs) atomicAdd(&dc->proj_macs, macs);
        }
    } else {
        // ---- split, drain, store
        // X: a warp takes rows (lane / 8) 4 + warp % 4 + 16 (warp / 4) + 64 u, eight lanes a row (rows 4 apart fall into
        // different halves of the swizzle).  W: a warp takes rows warp + 16 u of the step, a lane four columns.
        const int xrow = (lane >> 3) * 4 + (warp & 3) + 16 * (warp >> 2), xc = lane & 7;
        const uint32_t q = warp & 3, col0 = 32 * (warp >> 2);                 // rows and columns drained by this warp
        const uint32_t lanes = (q * 32) << 16;
        uint32_t g = 0, gc = 0, i = 0;
        bool ok = true;
        auto mark_of = [&](uint32_t tile) {             // (a mark stands for one tile but in very large calls)
            return tile / (((ntiles + gridDim.x - 1) / gridDim.x + FT_MARKS - 1) / FT_MARKS);
        };
        auto mark = [&]() { atomicOr(&marks[mark_of(i) / 32], 1u << (mark_of(i) % 32)); };
        // the stream of loads, two steps ahead of the splitting: tile, step, and where this thread stands in X and W
        float4 xv[2][2], wv[2][2];
        int lt = blockIdx.x, lk = 0;
        const float *px = nullptr, *pw = nullptr;
        bool x_in[2], w_in = false;
        auto aim = [&]() {
            const int r = lt / nt, m = (r % mt) * FT_M + xrow, n = (lt % nt) * FT_N + 4 * lane, w = r / mt;
            px = X + (size_t)m * K + 4 * xc;
            pw = (w == 0 ? W0 : (w == 1 ? W1 : W2)) + (size_t)warp * N + n;
            x_in[0] = m < M; x_in[1] = m + 64 < M;
            w_in = n < N;
        };
        const size_t x_half = (size_t)64 * K, w_half = (size_t)16 * N;
        auto load = [&](float4 (&x)[2], float4 (&w)[2]) {       // zeros outside the matrices
            if (lt >= ntiles) return;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                x[u] = x_in[u] && lk + 4 * xc < K ? __ldg(reinterpret_cast<const float4*>(px + u * x_half)) : zero;
                w[u] = w_in && lk + warp + 16 * u < K ? __ldg(reinterpret_cast<const float4*>(pw + u * w_half)) : zero;
            }
            px += FT_K;
            pw += (size_t)FT_K * N;
            lk += FT_K;
            if (lk >= nsteps * FT_K) { lk = 0; lt += gridDim.x; if (lt < ntiles) aim(); }
        };
        if (lt < ntiles) aim();
        load(xv[0], wv[0]);
        load(xv[1], wv[1]);
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
            float acc[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e] = 0.f;
            auto drain = [&](uint32_t src) {             // adds 32 columns of an accumulator to the running sums
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t v[16];
                    tmem_ld16(src + lanes + col0 + 16 * h, v);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[16 * h + e] += __uint_as_float(v[e]);
                }
                tc_fence_before();
                __syncwarp();
            };
            auto drain_main = [&]() -> bool {            // chunk gc
                if (!__all_sync(0xffffffffu, mbar_wait(&main_full[gc & 1], (gc >> 1) & 1, abortp))) return false;
                tc_fence_after();
                drain(tmem + FT_TMEM_MAIN + (gc & 1) * FT_N);
                if (lane == 0) mbar_arrive(&main_empty[gc & 1]);
                ++gc;
                return true;
            };
            auto step = [&](int s, float4 (&x)[2], float4 (&w)[2]) -> bool {
                const int slot = g % FT_SLOTS;
                if (g >= FT_SLOTS && !__all_sync(0xffffffffu, mbar_wait(&empty_bar[slot], ((g / FT_SLOTS) - 1) & 1, abortp))) return false;
                uint8_t* buf = smem + (slot >> 1) * FT_BUF_BYTES;
                uint32_t least = 0xffffffffu;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    ft_split_store(buf + swz128_offset(xrow + 64 * u, (slot & 1) * 4 + (xc >> 1)) + 8 * (xc & 1), x[u], least);
                    ft_split_store(buf + 3 * FT_PLANE_BYTES + (lane >> 4) * (FT_PLANE_BYTES / 2) +
                                       swz128_offset((slot & 1) * 32 + warp + 16 * u, (lane & 15) >> 1) + 8 * (lane & 1), w[u], least);
                }
                if (least < FT_SMALL) mark();
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_bar[slot]);
                ++g;
                load(x, w);
                // The chunk before this one is complete: its last step's slot has just been given back.
                return !(s % FT_CHUNK == FT_CHUNK - 1 && s >= 2 * FT_CHUNK - 1) || drain_main();
            };
            for (int s = 0; s < nsteps && ok; s += 2) ok = step(s, xv[0], wv[0]) && step(s + 1, xv[1], wv[1]);
            const uint32_t chunks = (nsteps + FT_CHUNK - 1) / FT_CHUNK;      // not drained yet: the last, and the one before if the last is short
            const uint32_t left = chunks - (nsteps >= 2 * FT_CHUNK ? (uint32_t)(nsteps / FT_CHUNK - 1) : 0u);
            for (uint32_t c = 0; c < left && ok; ++c) ok = drain_main();
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&cross_full, i & 1, abortp));
            if (ok) {
                tc_fence_after();
                drain(tmem + FT_TMEM_CROSS);
                if (lane == 0) mbar_arrive(&cross_empty);
                bool finite = true;
#pragma unroll
                for (int e = 0; e < 32; ++e) finite = finite && fabsf(acc[e]) < INFINITY;
                if (!finite) mark();
            }
            // (the warps leave together if one of them gave up a wait)
            ok = named_bar_all(ok, 1, 32 * FT_WORKERS);
            if (!ok) break;
            // every MMA of the tile is complete: the ring's first buffer stages the outputs, a warp's 32 rows x 32 columns on
            // their own, so that a row leaves as 128 consecutive bytes
            const int r = t / nt, m0 = (r % mt) * FT_M + 32 * q, n0 = (t % nt) * FT_N + col0, w = r / mt;
            float* O = w == 0 ? O0 : (w == 1 ? O1 : O2);
            float* stage = reinterpret_cast<float*>(smem) + warp * 32 * FT_PITCH;
#pragma unroll
            for (int e = 0; e < 32; e += 4)
                *reinterpret_cast<float4*>(stage + lane * FT_PITCH + e) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
            __syncwarp();
#pragma unroll 2
            for (int rr = lane >> 3; rr < 32; rr += 4) {
                const int m = m0 + rr, n = n0 + 4 * (lane & 7);
                if (m >= M || n >= N) continue;
                float4 y = *reinterpret_cast<const float4*>(stage + rr * FT_PITCH + 4 * (lane & 7));
                if (R) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(R + (size_t)m * N + n));
                    y.x += x.x; y.y += x.y; y.z += x.z; y.w += x.w;
                }
                *reinterpret_cast<float4*>(O + (size_t)m * N + n) = y;
            }
            named_bar_sync(1, 32 * FT_WORKERS);          // the staging area is an operand buffer again
        }
        // ---- tiles that were marked (outputs and marks of all warps are complete behind the last barrier)
        if (ok) {
            for (uint32_t j = 0; j < i; ++j) {
                if (!(marks[mark_of(j) / 32] >> (mark_of(j) % 32) & 1u)) continue;
                const int t = blockIdx.x + j * gridDim.x, r = t / nt, w = r / mt;
                ft_form_again<FT_WORKERS>(X, w == 0 ? W0 : (w == 1 ? W1 : W2), w == 0 ? O0 : (w == 1 ? O1 : O2), R, (r % mt) * FT_M, (t % nt) * FT_N, M, K,
                              N, reinterpret_cast<FtAgain*>(smem));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == FT_WORKERS) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------- operands split once, pairs of CTAs
// The largest calls: X and W are split into parts in global memory by a kernel of their own (the kernel above splits every tile
// of X once per column tile and every tile of W once per row tile, beside its MMAs), and the product is that of psa_gemm.cu's
// pairs of CTAs, 256 x 256 tiles, with six MMAs where that has one: per 64 k the five smaller products of all of them, then the
// leading ones into the same accumulator, which is read and added to the running sums in registers: no sum in the tensor core that
// has reached its size is longer than 4.
//
// What bounds it: 24 MMAs of 256 x 256 x 16 per 64 k, 3072 cycles of MMA, measured 5000 (the pairs of psa_gemm.cu take 160 cycles per MMA
// where 128 are nominal, and every 64 k an accumulator is handed over twice).  2048 x 768 x 3 x 768: 60 us on 128 x 128 tiles, 42 here with
// 7 of the split; the layer of 4 x 512 vectors 105 -> 85 us.
//
// Error against 64 bits (relative, 2-norm), the kernel above / this one: normal inputs, K = 320 / 768 / 2048 1.19 / 1.31 / 1.46e-7 and 0.91 /
// 1.04 / 1.32e-7; positive inputs, K = 768, 1.74e-7 and 0.99e-7.
constexpr int FP_BK = 64, FP_PLANE = 128 * FP_BK * 2;                       // a part of a CTA's operand: 16 KB
constexpr int FP_STAGE = 6 * FP_PLANE, FP_STAGES = 2, FP_WORKERS = 8, FP_THREADS = 64 + 32 * FP_WORKERS;
constexpr int FP_SMEM = FP_STAGES * FP_STAGE + 1024;
struct FPMaps {
    CUtensorMap a, b[3];      // parts as [3, rows, 1, columns]: boxes of 128 rows, of 64 rows x 64 columns
};
static_assert(sizeof(FtAgain) <= FP_STAGE, "does not fit the ring");

// blockIdx.y: 0 X, 1.. W.  Splits `count4` groups of four numbers and marks blocks of 128 rows of X, of 256 columns of W, in which
// a nonzero number is below 2^-60.
__global__ void __launch_bounds__(256)
f32_split_operands_kernel(const float4* __restrict__ X, const float4* W0, const float4* W1, const float4* W2, uint2* __restrict__ xp, uint2* __restrict__ wp,
                          uint32_t x4, uint32_t w4, uint32_t k4, uint32_t n4, int* __restrict__ x_small, int* __restrict__ w_small,
                          int mark) {
    const int which = blockIdx.y;
    const float4* src = which == 0 ? X : (which == 1 ? W0 : (which == 2 ? W1 : W2));
    const uint32_t count4 = which == 0 ? x4 : w4;
    grid_dependency_wait();
    uint2* dst = which == 0 ? xp : wp + (size_t)(which - 1) * 3 * w4;
    const int blocks_n = (int)((n4 + 63) / 64);
    for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < count4; i += gridDim.x * 256u) {
        const float4 v = __ldg(src + i);
        const float x[4] = {v.x, v.y, v.z, v.w};
        uint32_t p[3][4], least = 0xffffffffu;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            least = min(least, 2u * __float_as_uint(x[e]) - 1u);
            p[0][e] = (__float_as_uint(x[e]) + 0x8000u) & 0xffff0000u;
            const float r1 = x[e] - __uint_as_float(p[0][e]);
            p[1][e] = __float_as_uint(r1) & 0xffff0000u;
            p[2][e] = __float_as_uint(r1 - __uint_as_float(p[1][e]));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) dst[(size_t)k * count4 + i] = make_uint2(ft_pack(p[k][0], p[k][1]), ft_pack(p[k][2], p[k][3]));
        if (least < FT_SMALL) {
            if (which == 0) x_small[i / k4 / FT_M] = mark;
            else w_small[(which - 1) * blocks_n + (i % n4) / 64] = mark;
        }
    }
}

__global__ void __launch_bounds__(FP_THREADS, 1)
f32_project_pairs_kernel(const __grid_constant__ FPMaps maps, const float* __restrict__ X, const float* W0, const float* W1, const float* W2, float* O0,
                         float* O1, float* O2, int M, int K, int N, int nW, const float* __restrict__ R, const int* __restrict__ x_small,
                         const int* __restrict__ w_small, int mark, DeviceCounters* dc) {
    extern __shared__ uint8_t fp_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(fp_smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full_bar[FP_STAGES], empty_bar[FP_STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_flag;
    __shared__ uint32_t marks[FT_MARKS / 32];      // tiles of this CTA to look at again
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank(), unit = blockIdx.x / 2, units = gridDim.x / 2;
    const int nk = (K + FP_BK - 1) / FP_BK, mt = (M + 255) / 256, nt = (N + 255) / 256, ntiles = mt * nt * nW;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < FP_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * FP_WORKERS); }
        fence_mbar_init();
    }
    for (int i = threadIdx.x; i < FT_MARKS / 32; i += FP_THREADS) marks[i] = 0;
    if (warp == 1) { tmem_alloc_pair(&tmem_base_s, 512); tmem_relinquish_pair(); }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                                // the partner's barriers are initialised
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    volatile int* abortp = &abort_flag;
    grid_dependency_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: the two CTAs fill their halves of a stage, the first one's barrier collects the bytes of both
            int g = 0;
            bool ok = true;
            for (int t = unit; t < ntiles && ok; t += units) {
                const int r = t / nt, w = r / mt, m0 = (r % mt) * 256 + rank * 128, n0 = (t % nt) * 256 + rank * 128;
                for (int kt = 0; kt < nk; ++kt, ++g) {
                    const int s = g % FP_STAGES;
                    if (g >= FP_STAGES && !mbar_wait(&empty_bar[s], ((g / FP_STAGES) - 1) & 1, abortp)) { ok = false; break; }
                    uint8_t* st = smem + s * FP_STAGE;
                    if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 2 * FP_STAGE);
                    const uint32_t bar = cluster_map(&full_bar[s], 0);
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        tma_load_4d_pair(st + p * FP_PLANE, &maps.a, bar, kt * FP_BK, 0, m0, p);
                        tma_load_4d_pair(st + (3 + p) * FP_PLANE, &maps.b[w], bar, n0, 0, kt * FP_BK, p);
                        tma_load_4d_pair(st + (3 + p) * FP_PLANE + FP_PLANE / 2, &maps.b[w], bar, n0 + 64, 0, kt * FP_BK, p);
                    }
                }
            }
            if (*abortp && rank == 0)
                for (int k = max(0, g - FP_STAGES); k < g; ++k) mbar_wait_drain(&full_bar[k % FP_STAGES], (k / FP_STAGES) & 1);
        }
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {
            // ---- MMA issuer
            const uint32_t idesc = umma_idesc_bf16(256, 256, UMMA_K_MAJOR, UMMA_MN_MAJOR);
            const uint32_t a_lo0 = umma_desc_lo_kmajor(smem_u32(smem)), b_lo0 = umma_desc_lo_mnmajor(smem_u32(smem + 3 * FP_PLANE), FP_PLANE / 2);
            constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};      // the leading product last
            unsigned long long macs = 0;
            int g = 0;
            bool ok = true;
            for (int t = unit; t < ntiles && ok; t += units) {
                for (int kt = 0; kt < nk; ++kt, ++g) {
                    const int s = g % FP_STAGES, buf = g & 1;
                    if (g >= 2) ok = mbar_wait(&acc_empty[buf], ((g >> 1) - 1) & 1, abortp);
                    if (ok) ok = mbar_wait(&full_bar[s], (g / FP_STAGES) & 1, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = a_lo0 + s * (FP_STAGE >> 4), b = b_lo0 + s * (FP_STAGE >> 4);
#pragma unroll
                    for (int q = 0; q < 6; ++q)
#pragma unroll
                        for (int k = 0; k < FP_BK / 16; ++k)
                            umma_ss_pair(tmem + buf * 256, umma_desc_join(a + ((PA[q] * FP_PLANE + k * 32) >> 4), UMMA_DESC_HI_SW128),
                                         umma_desc_join(b + ((PB[q] * FP_PLANE + k * 2048) >> 4), UMMA_DESC_HI_SW128), idesc, q != 0 || k != 0);
                    umma_commit_pair(&empty_bar[s]);
                    umma_commit_pair(&acc_full[buf]);
                }
                const int r = t / nt;
                if (ok) macs += (unsigned long long)min(256, M - (r % mt) * 256) * min(256, N - (t % nt) * 256) * K;
            }
            if (macs) atomicAdd(&dc->proj_macs, macs);
        }
    } else {
        // ---- running sums: a warp has 32 rows (TMEM lanes) by 128 columns
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t src0 = tmem + (static_cast<uint32_t>(q * 32) << 16) + half * 128;
        const uint32_t empty0 = cluster_map(&acc_empty[0], 0), empty1 = cluster_map(&acc_empty[1], 0);
        int g = 0, i = 0;
        bool ok = true;
        auto mark_of = [&](int tile) { return tile / (((ntiles + units - 1) / units + FT_MARKS - 1) / FT_MARKS); };
        for (int t = unit; t < ntiles && ok; t += units, ++i) {
            float acc[128];
#pragma unroll
            for (int e = 0; e < 128; ++e) acc[e] = 0.f;
            for (int kt = 0; kt < nk; ++kt, ++g) {
                const int buf = g & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (g >> 1) & 1, abortp));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    uint32_t v[16];
                    tmem_ld16(src0 + buf * 256 + 16 * u, v);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[16 * u + e] += __uint_as_float(v[e]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(buf ? empty1 : empty0);
            }
            if (!ok) break;
            const int r = t / nt, w = r / mt, m0 = (r % mt) * 256 + rank * 128, n0 = (t % nt) * 256 + half * 128, row = m0 + 32 * q + lane;
            float* o = (w == 0 ? O0 : (w == 1 ? O1 : O2)) + (size_t)row * N + n0;
            if (row < M) {
                bool finite = true;
#pragma unroll
                for (int e = 0; e < 128; e += 4) {
                    if (n0 + e < N) {
                        finite = finite && fabsf(acc[e]) < INFINITY && fabsf(acc[e + 1]) < INFINITY && fabsf(acc[e + 2]) < INFINITY && fabsf(acc[e + 3]) < INFINITY;
                        float4 y = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
                        if (R) {
                            const float4 x = __ldg(reinterpret_cast<const float4*>(R + (size_t)row * N + n0 + e));
                            y.x += x.x; y.y += x.y; y.z += x.z; y.w += x.w;
                        }
                        *reinterpret_cast<float4*>(o + e) = y;
                    }
                }
                if (!finite || x_small[m0 / FT_M] == mark || w_small[w * nt + t % nt] == mark) atomicOr(&marks[mark_of(i) / 32], 1u << (mark_of(i) % 32));
            }
        }
        // ---- tiles that were marked
        ok = named_bar_all(ok, 1, 32 * FP_WORKERS);
        if (ok)
            for (int j = 0; j < i; ++j) {
                if (!(marks[mark_of(j) / 32] >> (mark_of(j) % 32) & 1u)) continue;
                const int t = unit + j * units, r = t / nt, w = r / mt;
                for (int c = 0; c < 256; c += FT_N)
                    ft_form_again<FP_WORKERS>(X, w == 0 ? W0 : (w == 1 ? W1 : W2), w == 0 ? O0 : (w == 1 ? O1 : O2), R, (r % mt) * 256 + rank * 128,
                                              (t % nt) * 256 + c, M, K, N, reinterpret_cast<FtAgain*>(smem));
            }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    __syncwarp();
    cluster_sync();                 // MMAs, arrivals and copies that involve the partner are over in both CTAs
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

}  // namespace

cudaError_t f32_project_tensor(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D, int N,
                               const float* residual, DeviceCounters* dc, cudaStream_t stream) {
    static DeviceSetup setup;
    const int sms = device_setup(&setup, [] {
        return cudaFuncSetAttribute(f32_project_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FT_SMEM);
    }, "fp32 projection set-up");
    if (sms <= 0) return cudaErrorUnknown;
    const long long tiles = (long long)((rows + FT_M - 1) / FT_M) * ((N + FT_N - 1) / FT_N) * nW;
    f32_project_tensor_kernel<<<(int)(tiles < sms ? tiles : sms), FT_THREADS, FT_SMEM, stream>>>(
        X, W[0], W[nW == 3 ? 1 : 0], W[nW == 3 ? 2 : 0], out[0], out[nW == 3 ? 1 : 0], out[nW == 3 ? 2 : 0], rows, D, N, nW, residual, dc);
    return cudaGetLastError();
}

// Whether the pairs are faster, in cycles as measured: the split and 5000 per 64 k of a 256 x 256 tile against 2300 per 32 k of a 128 x 128
// tile of the kernel above (us, layers of 12 heads with d_model = 768: 1024 rows 65 / 58 on the tiles, 2048 rows 88 / 107).
bool f32_project_pairs_pay(int rows, int D, int N, int nW, int sms) {
    const long long pairs = (long long)((rows + 255) / 256) * ((N + 255) / 256) * nW, tiles = (long long)((rows + 127) / 128) * ((N + 127) / 128) * nW;
    const long long units = sms / 2 > 0 ? sms / 2 : 1;
    return 16000 + (pairs + units - 1) / units * ((D + 63) / 64) * 5000 < 4000 + (tiles + sms - 1) / sms * ((D + 31) / 32) * 2300;
}

cudaError_t f32_project_pairs(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D, int N, const float* residual,
                              void* parts, int* marks, int mark, DeviceCounters* dc, cudaStream_t stream) {
    static DeviceSetup setup;
    const int sms = device_setup(&setup, [] {
        return cudaFuncSetAttribute(f32_project_pairs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FP_SMEM);
    }, "fp32 projection set-up (pairs)");
    if (sms < 2) return cudaErrorUnknown;
    char* xp = static_cast<char*>(parts);
    char* wp = xp + ((size_t)rows * D * 6 + 255) / 256 * 256;
    const uint32_t x4 = (uint32_t)((size_t)rows * D / 4), w4 = (uint32_t)((size_t)D * N / 4);
    int* w_small = marks + (rows + 127) / 128;
    const uint32_t blocks = (max(x4, w4) + 1023) / 1024;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernels wait for their predecessors themselves
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t split = {};
    split.gridDim = dim3(blocks < 1024 ? blocks : 1024, 1 + nW);
    split.blockDim = dim3(256);
    split.stream = stream;
    split.attrs = attr;
    split.numAttrs = 1;
    const auto f4 = [&](int w) { return reinterpret_cast<const float4*>(W[nW == 3 ? w : 0]); };
    const cudaError_t e = cudaLaunchKernelEx(&split, f32_split_operands_kernel, reinterpret_cast<const float4*>(X), f4(0), f4(1), f4(2),
                                             reinterpret_cast<uint2*>(xp), reinterpret_cast<uint2*>(wp), x4, w4, (uint32_t)(D / 4), (uint32_t)(N / 4), marks, w_small, mark);
    if (e != cudaSuccess) return e;
    FPMaps maps;
    if (!make_tensor_map_bf16_4d(&maps.a, xp, 3, rows, 1, D, 128)) return cudaErrorInvalidValue;
    for (int w = 0; w < 3; ++w)
        if (!make_tensor_map_bf16_4d(&maps.b[w], wp + (size_t)(w < nW ? w : 0) * 6 * D * N, 3, D, 1, N, FP_BK)) return cudaErrorInvalidValue;
    const int ntiles = ((rows + 255) / 256) * ((N + 255) / 256) * nW, units = ntiles < sms / 2 ? ntiles : sms / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * units);
    cfg.blockDim = dim3(FP_THREADS);
    cfg.dynamicSmemBytes = FP_SMEM;
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, f32_project_pairs_kernel, maps, X, W[0], W[nW == 3 ? 1 : 0], W[nW == 3 ? 2 : 0], out[0], out[nW == 3 ? 1 : 0],
                              out[nW == 3 ? 2 : 0], rows, D, N, nW, residual, static_cast<const int*>(marks), static_cast<const int*>(w_small), mark, dc);
}

}  // namespace psa
