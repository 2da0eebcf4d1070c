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
// A CTA takes tiles of 128 x 128.  Warps 0-15 read X and W (two steps of 32 k ahead, in registers), split them into parts
// and write these as operand tiles in the 128-byte swizzle (X K-major, W MN-major) into a ring of four steps; warp 16
// issues 12 MMAs of 128 x 128 x 16 per step; warps 0-15 also drain the accumulators, 32 rows by 32 columns each.
//
// What bounds it: 12 MMAs per step at 92 cycles (N = 128) are 1104 cycles for 32 k; splitting a step takes about 600 issue
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
// What it costs, in a layer of 4 x 512 vectors, d_model = 768, 12 heads, of whose 176 us the projection takes 60: one 1e-35 in
// every vector, so that every tile is looked at, 208 us; nothing but numbers around 1e-33, so that every output is formed
// again, 439; nothing but NaN 416 (as a loop of one thread per 32 outputs in global memory it was 3300 in all three).
#include "psa_internal.h"
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

// Replaces those outputs of a finished tile that the parts cannot carry, by the plain chain: called by all FT_WORKERS warps.  A
// thread has the eight rows row0 + 4 i and the four columns from col0 on.  Without a residual the outputs say whether there is
// anything to replace; with one the tile is computed again in any case.
__device__ __noinline__ void ft_form_again(const float* X, const float* W, float* O, const float* R, int m_first, int n_first, int M, int K,
                                           int N, FtAgain* sm) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row0 = 32 * (warp & 3) + (lane >> 3), col0 = 32 * (warp >> 2) + 4 * (lane & 7);
    named_bar_sync(1, 32 * FT_WORKERS);       // (the tile before is done with the shared memory)
    if (tid < FT_M) { sm->row_least[tid] = sm->col_least[tid] = 0xffffffffu; sm->row_most[tid] = sm->col_most[tid] = 0; }
    named_bar_sync(1, 32 * FT_WORKERS);
    for (int r = warp; r < FT_M && m_first + r < M; r += FT_WORKERS) {
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
    if (n_first + 4 * lane < N) {
        uint32_t least[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu}, most[4] = {0, 0, 0, 0};
#pragma unroll 8
        for (int k = warp; k < K; k += FT_WORKERS) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(W + (size_t)k * N + n_first + 4 * lane));
            const uint32_t t[4] = {2u * __float_as_uint(v.x), 2u * __float_as_uint(v.y), 2u * __float_as_uint(v.z), 2u * __float_as_uint(v.w)};
#pragma unroll
            for (int e = 0; e < 4; ++e) { least[e] = min(least[e], t[e] - 1u); most[e] = max(most[e], t[e]); }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) { atomicMin(&sm->col_least[4 * lane + e], least[e]); atomicMax(&sm->col_most[4 * lane + e], most[e]); }
    }
    named_bar_sync(1, 32 * FT_WORKERS);
    const bool inside = n_first + col0 < N;                 // (N is a multiple of 4)
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
        for (int i = 0; i < 8; ++i) {
            if (!inside || m_first + row0 + 4 * i >= M) continue;
            const float4 o = *reinterpret_cast<const float4*>(out + (size_t)(4 * i) * N);
            any = any || lost(o.x, row0 + 4 * i, col0) || lost(o.y, row0 + 4 * i, col0 + 1) || lost(o.z, row0 + 4 * i, col0 + 2) ||
                  lost(o.w, row0 + 4 * i, col0 + 3);
        }
        if (named_bar_all(!any, 1, 32 * FT_WORKERS)) return;
    }
    float acc[8][4] = {};
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += FT_K) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 xv[2], wv[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = tid + 32 * FT_WORKERS * u, m = m_first + (t >> 3), kx = k0 + 4 * (t & 7), kw = k0 + (t >> 5), n = n_first + 4 * (t & 31);
            xv[u] = m < M && kx < K ? __ldg(reinterpret_cast<const float4*>(X + (size_t)m * K + kx)) : zero;
            wv[u] = kw < K && n < N ? __ldg(reinterpret_cast<const float4*>(W + (size_t)kw * N + n)) : zero;
        }
        named_bar_sync(1, 32 * FT_WORKERS);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = tid + 32 * FT_WORKERS * u;
            *reinterpret_cast<float4*>(sm->x + (t >> 3) * (FT_K + 4) + 4 * (t & 7)) = xv[u];
            *reinterpret_cast<float4*>(sm->w + 4 * t) = wv[u];
        }
        named_bar_sync(1, 32 * FT_WORKERS);
        const int kn = min(FT_K, K - k0);     // (a multiple of 4)
#pragma unroll 1
        for (int k = 0; k < kn; k += 4) {
            float4 w[4];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) w[kk] = *reinterpret_cast<const float4*>(sm->w + (k + kk) * FT_N + col0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(sm->x + (row0 + 4 * i) * (FT_K + 4) + k);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float f = kk == 0 ? x.x : kk == 1 ? x.y : kk == 2 ? x.z : x.w;
                    acc[i][0] = fmaf(f, w[kk].x, acc[i][0]); acc[i][1] = fmaf(f, w[kk].y, acc[i][1]);
                    acc[i][2] = fmaf(f, w[kk].z, acc[i][2]); acc[i][3] = fmaf(f, w[kk].w, acc[i][3]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = row0 + 4 * i;
        if (!inside || m_first + r >= M) continue;
        const size_t at = (size_t)(4 * i) * N;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float o = out[at + e];
            if (!(fabsf(o) < INFINITY) || lost(R ? acc[i][e] : o, r, col0 + e))
                out[at + e] = R ? acc[i][e] + R[(size_t)(m_first + r) * N + n_first + col0 + e] : acc[i][e];
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
                ft_form_again(X, w == 0 ? W0 : (w == 1 ? W1 : W2), w == 0 ? O0 : (w == 1 ? O1 : O2), R, (r % mt) * FT_M, (t % nt) * FT_N, M, K,
                              N, reinterpret_cast<FtAgain*>(smem));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(&dc->status, (int)PSA_ERR_TIMEOUT);
    if (warp == FT_WORKERS) tmem_dealloc(tmem, 512);
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

}  // namespace psa
