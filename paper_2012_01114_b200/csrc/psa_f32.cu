// The full-precision path: fp32 storage, and fp32 arithmetic on CUDA cores but for large calls, whose projections are in
// psa_f32_tensor.cu and whose attention (FULL, MASKED) is in psa_f32_attn_tensor.cu.  Skipping is element-exact: a weight that the
// scheme does not need is never computed (paper Sec. 4.1, 5.1), so issued MACs equal the paper's element counts (Sec. 3.2, 4.2,
// 5.2).  The throughput path is the bf16 one.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_ws.h"
#include "sm100.cuh"

namespace psa {

namespace {

constexpr int PROJ_TILE = 16;

// out[w][r, c] = sum_k X[r, k] W[w][k, c]      (paper Sec. 3.1: the projections are plain products)
__global__ void __launch_bounds__(PROJ_TILE* PROJ_TILE)
f32_project_kernel(const float* __restrict__ X, const float* W0, const float* W1, const float* W2, float* O0,
                   float* O1, float* O2, int rows, int D, int N, const float* __restrict__ R, DeviceCounters* dc) {
    __shared__ float xs[PROJ_TILE][PROJ_TILE + 1];
    __shared__ float ws[PROJ_TILE][PROJ_TILE + 1];
    const float* W = blockIdx.z == 0 ? W0 : (blockIdx.z == 1 ? W1 : W2);
    float* O = blockIdx.z == 0 ? O0 : (blockIdx.z == 1 ? O1 : O2);
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int r = blockIdx.y * PROJ_TILE + ty, c = blockIdx.x * PROJ_TILE + tx;
    float acc = 0.f;
    for (int k0 = 0; k0 < D; k0 += PROJ_TILE) {
        xs[ty][tx] = (r < rows && k0 + tx < D) ? X[(size_t)r * D + k0 + tx] : 0.f;
        ws[ty][tx] = (k0 + ty < D && c < N) ? W[(size_t)(k0 + ty) * N + c] : 0.f;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PROJ_TILE; ++k) acc = fmaf(xs[ty][k], ws[k][tx], acc);
        __syncthreads();
    }
    if (r < rows && c < N) O[(size_t)r * N + c] = R ? acc + R[(size_t)r * N + c] : acc;
    if (tx == 0 && ty == 0) {
        const int vr = min(PROJ_TILE, rows - blockIdx.y * PROJ_TILE), vc = min(PROJ_TILE, N - blockIdx.x * PROJ_TILE);
        atomicAdd(&dc->proj_macs, (unsigned long long)vr * vc * D);
    }
}

// ---------------------------------------------------------------- tiled kernels
// Two fp32 multiply-accumulates in one instruction, each rounded as fmaf rounds it.
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float v) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
// Asynchronous copies global -> shared (4 and 16 bytes) and the waits for them.
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Projection of small calls on CUDA cores: 32 x 32 outputs per CTA of 128 threads, two rows 16 apart by four columns per
// thread, operands staged GP_STAGES deep with asynchronous copies.  Every output is the same chain of fmaf over k = 0, 1, ...
// as in f32_project_kernel, so the results are bitwise the same.  Needs D and N to be multiples of 4.  Bound by the latency of
// its k-steps: 768 deep, 16 ... 256 rows take 23-30 us.
constexpr int GP_BM = 32, GP_BN = 32, GP_TM = 2, GP_BK = 32, GP_LDA = GP_BK + 4, GP_STAGES = 3;
constexpr int GP_TX = GP_BN / 4, GP_TY = GP_BM / GP_TM, GP_THREADS = GP_TX * GP_TY;
constexpr int GP_A_FLOATS = GP_BM * GP_LDA, GP_STAGE = GP_A_FLOATS + GP_BK * GP_BN;
constexpr int GP_SMEM = GP_STAGES * GP_STAGE * (int)sizeof(float);

__global__ void __launch_bounds__(GP_THREADS)
f32_project_tiled_kernel(const float* __restrict__ X, const float* W0, const float* W1, const float* W2, float* O0,
                         float* O1, float* O2, int rows, int D, int N, const float* __restrict__ R, DeviceCounters* dc) {
    extern __shared__ float4 gp_smem4[];
    float* sm = reinterpret_cast<float*>(gp_smem4);
    const float* W = blockIdx.z == 0 ? W0 : (blockIdx.z == 1 ? W1 : W2);
    float* O = blockIdx.z == 0 ? O0 : (blockIdx.z == 1 ? O1 : O2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tx = lane & 7, ty = warp * 4 + (lane >> 3);
    const int m0 = blockIdx.y * GP_BM, n0 = blockIdx.x * GP_BN;
    const int nk = (D + GP_BK - 1) / GP_BK;

    auto load = [&](int kt) {       // k-step kt; what lies outside the matrices is not loaded, and nothing that is stored reads it
        float* a = sm + (kt % GP_STAGES) * GP_STAGE;
        float* b = a + GP_A_FLOATS;
        const int k0 = kt * GP_BK;
        for (int t = tid; t < GP_BM * (GP_BK / 4); t += GP_THREADS) {
            const int r = t / (GP_BK / 4), c = (t % (GP_BK / 4)) * 4;
            if (m0 + r < rows && k0 + c < D) cp_async16(a + r * GP_LDA + c, X + (size_t)(m0 + r) * D + k0 + c);
        }
        for (int t = tid; t < GP_BK * (GP_BN / 4); t += GP_THREADS) {
            const int k = t / (GP_BN / 4), c = (t % (GP_BN / 4)) * 4;
            if (n0 + c < N && k0 + k < D) cp_async16(b + k * GP_BN + c, W + (size_t)(k0 + k) * N + n0 + c);
        }
    };
    unsigned long long acc[GP_TM][2] = {};
#pragma unroll
    for (int s = 0; s < GP_STAGES - 1; ++s) {
        if (s < nk) load(s);
        cp_async_commit();
    }
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait_group<GP_STAGES - 2>();
        __syncthreads();            // step kt has landed, and step kt - 1's buffer is free
        if (kt + GP_STAGES - 1 < nk) load(kt + GP_STAGES - 1);
        cp_async_commit();
        const float* a = sm + (kt % GP_STAGES) * GP_STAGE + ty * GP_LDA;
        const float* b = sm + (kt % GP_STAGES) * GP_STAGE + GP_A_FLOATS + 4 * tx;
        const int kn = min(GP_BK, D - kt * GP_BK);
#pragma unroll 2
        for (int k = 0; k < kn; k += 4) {
            float4 av[GP_TM];
#pragma unroll
            for (int i = 0; i < GP_TM; ++i) av[i] = *reinterpret_cast<const float4*>(a + i * GP_TY * GP_LDA + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const ulonglong2 bv = *reinterpret_cast<const ulonglong2*>(b + (k + kk) * GP_BN);
#pragma unroll
                for (int i = 0; i < GP_TM; ++i) {
                    const unsigned long long x = dup2(kk == 0 ? av[i].x : kk == 1 ? av[i].y : kk == 2 ? av[i].z : av[i].w);
                    fma2(acc[i][0], x, bv.x);
                    fma2(acc[i][1], x, bv.y);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < GP_TM; ++i) {
        const int r = m0 + ty + i * GP_TY;
        if (r >= rows) continue;
        const int c = n0 + 4 * tx;
        if (c >= N) continue;
        const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
        float4 o = make_float4(lo.x, lo.y, hi.x, hi.y);
        if (R) {
            const float4 x = *reinterpret_cast<const float4*>(R + (size_t)r * N + c);
            o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
        }
        *reinterpret_cast<float4*>(O + (size_t)r * N + c) = o;
    }
    if (tid == 0)
        atomicAdd(&dc->proj_macs, (unsigned long long)min(GP_BM, rows - m0) * min(GP_BN, N - n0) * D);
}

// Attention, tiled: a CTA of four warps works on BR = 64 / KS query rows of one (batch, head) and walks the keys in
// blocks of 64 staged in shared memory.  A warp owns 16 rows and 64 / KS keys of every block: two half-warps of 16
// lanes, lane (ty, tx) holding rows ty + 2 i (i < 8) and keys tx + 16 u (u < 4 / KS) of S, and output columns 4 tx .. + 3
// (and 64 + 4 tx .. + 3).  With KS > 1 the KS warps of a row group see different keys of each block and are merged
// once at the end.
//
// Element-exact skipping: lim_i is the last key of the warp's share that row i keeps; groups of 16 keys that a whole
// warp keeps run without tests, groups that nobody keeps are passed over, the rest is predicated weight by weight.  The
// same limits bound phase 3.
//
// What bounds it: the fp32 pipe (100-105 multiply-accumulates per clock and SM measured in chains, 128 nominal) and, level with
// it, instruction issue: phase 1 pairs components in two-wide fma, which leaves issue slots to its loads; phase 3 would have to
// double every weight into a pair and runs on plain fma.  Measured (us, one warp per row before): 48 heads of n = 512, d = 64,
// full 1554 -> 117; 16 heads of n = 1024, d = 128, masked 2003 -> 172; in a large call 61 multiply-accumulates per clock and SM.
// (DG = 1 is compiled for three CTAs per SM, 168 registers; with KS = 1 it spills 128 bytes there.)
//
// Shared memory, so that no address needs arithmetic in the inner loops: K rows are padded by 16 bytes (16 rows are read at
// once), Q rows keep 16-byte chunk c at c ^ (row & 1) (rows of both half-warps are read at once), V rows are plain.
constexpr int FA_THREADS = 128, FA_BC = 64;

template <int DG, int KS>
struct FACfg {
    static constexpr int DP = 64 * DG, KP = DP + 4;                     // row pitches of Q and V, of K, in floats
    static constexpr int BR = 64 / KS, U = 4 / KS, KW = FA_BC / KS;     // rows per CTA; key groups and keys of a warp
    static constexpr int PP = KW % 32 == 0 && !(DG == 2 && KS == 1) ? KW + 16 : KW;    // row pitch of P (the exception: room for two CTAs)
    static constexpr int Q_FLOATS = BR * DP, K_FLOATS = FA_BC * KP, V_FLOATS = FA_BC * DP, P_FLOATS = 4 * 16 * PP;
    static constexpr int SMEM = (Q_FLOATS + K_FLOATS + V_FLOATS + P_FLOATS) * (int)sizeof(float);
};

// Rows r0 .. r0 + ROWS - 1 of one head into a tile of row pitch PITCH (rows beyond n stay as they are; nothing reads them).
template <int DG, int ROWS, int PITCH, bool SWAP>
__device__ __forceinline__ void fa_load(float* tile, const float* src, int r0, int n, size_t ld, int d4) {
    const int c = threadIdx.x % (16 * DG), r = threadIdx.x / (16 * DG);
    constexpr int STEP = FA_THREADS / (16 * DG);
    if (c >= d4) return;
    const float* p = src + (size_t)(r0 + r) * ld + 4 * c;
    float* dst = tile + r * PITCH;
#pragma unroll
    for (int k = 0; k < ROWS / STEP; ++k) {
        if (r0 + r + k * STEP < n) cp_async16(dst + k * STEP * PITCH + 4 * (SWAP ? c ^ ((r + k * STEP) & 1) : c), p + (size_t)(k * STEP) * ld);
    }
}

// acc[i][u] += q_i . k_u, sums of even and odd components side by side.  q: row ty of the warp's rows, k: row tx of its keys.
// EDGE: only the weights that are kept.
template <int DG, int U, bool EDGE>
__device__ __forceinline__ void fa_scores(unsigned long long (&acc)[8][U], const float* q, const float* k, int d4, int tx, int ty,
                                          const int (&lim)[8], int minlim, int maxlim) {
    constexpr int DP = 64 * DG, KP = DP + 4;
    auto step = [&](const float* qc, const float* kc) {
        ulonglong2 kv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) kv[u] = *reinterpret_cast<const ulonglong2*>(kc + 16 * u * KP);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(qc + 2 * i * DP);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (EDGE) {
                    if (16 * u > maxlim) continue;                                  // (same for the whole warp)
                    if (16 * u + 15 > minlim && tx + 16 * u > lim[i]) continue;
                }
                fma2(acc[i][u], qv.x, kv[u].x);
                fma2(acc[i][u], qv.y, kv[u].y);
            }
        }
    };
    const float* qe = q + 4 * ty;           // chunks of even number of this lane's rows, and of odd number
    const float* qo = q - 4 * ty;
    int c = 0;
#pragma unroll 1
    for (; c + 1 < d4; c += 2) {
        step(qe + 4 * c, k + 4 * c);
        step(qo + 4 * c + 4, k + 4 * c + 4);
    }
    if (c < d4) step(qe + 4 * c, k + 4 * c);
}

// MODE 0: the three phases for FULL / MASKED.  MODE 2: phases 2 and 3 of the symmetric scheme, scores read from S.
// `bad` (may be null): MODE 0 works on the heads marked there only.
template <int DG, int KS, int MODE>
__global__ void __launch_bounds__(FA_THREADS, DG == 1 ? 3 : 2)
f32_flash_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V,
                 float* __restrict__ out, const float* __restrict__ S, int n, int H, int d, float scale, int masked,
                 DeviceCounters* dc, DeviceCounters* dc_next, const int* __restrict__ bad, int mark) {
    using C = FACfg<DG, KS>;
    constexpr int U = C::U;
    extern __shared__ float4 fa_smem4[];
    float* Qs = reinterpret_cast<float*>(fa_smem4);
    float* Ks = Qs + C::Q_FLOATS;
    float* Vs = Ks + C::K_FLOATS;
    float* Ps = Vs + C::V_FLOATS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tx = lane & 15, ty = lane >> 4;
    const int bh = blockIdx.x, b = bh / H, h = bh - b * H;
    if (MODE == 0) grid_dependency_wait();
    // the counter block of the NEXT call on this workspace is cleared here, off that call's critical path
    if (dc_next && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *dc_next = DeviceCounters{0, 0, 0, 0, 0, 0, 0};
    if (MODE == 0) {
        if (bad && bad[bh] != mark) return;
    }
    const int rb = masked ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;   // the longest rows first
    const int r0 = rb * C::BR;
    const int rg = warp / KS, kw = (warp % KS) * C::KW;                 // the warp's row group and first key of a block
    const int qrow = 16 * rg + ty, row = r0 + qrow;                     // row i of the lane: + 2 i
    const int wr0 = r0 + 16 * rg;                                       // first row of the warp
    const size_t ld = (size_t)H * d;
    const size_t base = ((size_t)b * n) * ld + (size_t)h * d;
    const int d4 = d >> 2;
    const int kend = masked ? min(r0 + C::BR, n) : n;                   // keys that some row of the CTA keeps
    const int nblk = (kend + FA_BC - 1) / FA_BC;
    const float* Sh = MODE == 2 ? S + (size_t)bh * n * n : nullptr;
    float* Pw = Ps + warp * 16 * C::PP;
    const float* Pr = Pw + ty * C::PP;                                  // row i of the lane: + 2 i PP
    const float* vb = Vs + kw * C::DP + 4 * tx;
    const bool act0 = tx < d4, act1 = DG == 2 && 16 + tx < d4;          // output columns this lane owns

    if (MODE != 2) {
        fa_load<DG, C::BR, C::DP, true>(Qs, Q + base, r0, n, ld, d4);
        fa_load<DG, FA_BC, C::KP, false>(Ks, K + base, 0, n, ld, d4);
    }
    cp_async_commit();

    float m[8], l[8], o[8][4 * DG];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
        for (int g = 0; g < 4 * DG; ++g) o[i][g] = 0.f;
    }
    unsigned int dots = 0, wts = 0;                                     // weights of this lane; of its rows in phase 3

    for (int jb = 0; jb < nblk; ++jb) {
        const int k0 = jb * FA_BC + kw;                                 // first key of the warp's share
        const int last = min(wr0 + 15, n - 1);                          // last row of the warp that exists
        const int maxlim = wr0 >= n ? -1 : (masked ? last : n - 1) - k0;
        const int minlim = wr0 + 15 >= n ? -1 : (masked ? wr0 : n - 1) - k0;

        if (MODE != 2) cp_async_wait_all();
        __syncthreads();            // K_j has landed; every warp is done with V_{j-1}
        fa_load<DG, FA_BC, C::DP, false>(Vs, V + base, jb * FA_BC, n, ld, d4);
        cp_async_commit();
        auto block = [&](auto edge_tag) {
            constexpr bool EDGE = decltype(edge_tag)::value;
            int lim[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) lim[i] = !EDGE ? C::KW - 1 : row + 2 * i >= n ? -1 : min(masked ? row + 2 * i : n - 1, n - 1) - k0;
            float s[8][U];
            // ---- phase 1 (Eq. 1)
            if (MODE == 2) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        s[i][u] = !EDGE || tx + 16 * u <= lim[i] ? __ldg(Sh + (size_t)(row + 2 * i) * n + k0 + tx + 16 * u) : -INFINITY;
            } else {
                unsigned long long acc[8][U] = {};
                if (!EDGE || maxlim >= 0)
                    fa_scores<DG, U, EDGE>(acc, Qs + qrow * C::DP, Ks + (kw + tx) * C::KP, d4, tx, ty, lim, minlim, maxlim);
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float2 f = unpack2(acc[i][u]);
                        s[i][u] = (f.x + f.y) * scale;
                        if (EDGE) {
                            const bool keep = tx + 16 * u <= lim[i];
                            s[i][u] = keep ? s[i][u] : -INFINITY;
                            dots += keep;
                        }
                    }
                if (!EDGE) dots += 8 * U;
            }
            // ---- phase 2 (Eq. 2): running row maximum and sum; the sum stays per lane until the end
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float mx = s[i][0];
#pragma unroll
                for (int u = 1; u < U; ++u) mx = fmaxf(mx, s[i][u]);
#pragma unroll
                for (int off = 8; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                mx = fmaxf(mx, m[i]);
                const float sub = mx == -INFINITY ? 0.f : mx;           // (no finite score yet: every weight is 0)
                if (mx != m[i]) {
                    const float alpha = expf(m[i] - mx);
                    m[i] = mx;
                    l[i] *= alpha;
#pragma unroll
                    for (int g = 0; g < 4 * DG; ++g) o[i][g] *= alpha;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!EDGE || tx + 16 * u <= lim[i]) {
                        const float e = expf(s[i][u] - sub);
                        l[i] += e;
                        Pw[(ty + 2 * i) * C::PP + tx + 16 * u] = e;
                    }
                }
                if (EDGE && tx == 0) wts += min(max(lim[i] + 1, 0), C::KW);
            }
            if (!EDGE && tx == 0) wts += 8 * C::KW;
        };
        const bool whole = minlim >= C::KW - 1;
        if (whole) block(std::false_type{});
        else block(std::true_type{});
        cp_async_wait_all();
        __syncthreads();            // V_j has landed, P is written; every warp is done with K_j
        if (MODE != 2 && jb + 1 < nblk) fa_load<DG, FA_BC, C::KP, false>(Ks, K + base, (jb + 1) * FA_BC, n, ld, d4);
        cp_async_commit();
        // ---- phase 3 (Eq. 3): keys in order, the warp's columns of V against its weights
        if (act0) {
            const int jfull = whole ? C::KW : (minlim + 1 > 0 ? (minlim + 1) & ~3 : 0);
            const float* pj = Pr;
            const float* vj = vb;
#pragma unroll 1
            for (int j = 0; j < jfull; j += 4, pj += 4, vj += 4 * C::DP) {
                float4 p[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) p[i] = *reinterpret_cast<const float4*>(pj + 2 * i * C::PP);
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const float4 v0 = *reinterpret_cast<const float4*>(vj + jj * C::DP);
                    float4 v1 = v0;
                    if (DG == 2 && act1) v1 = *reinterpret_cast<const float4*>(vj + jj * C::DP + 64);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float w = jj == 0 ? p[i].x : jj == 1 ? p[i].y : jj == 2 ? p[i].z : p[i].w;
                        o[i][0] = fmaf(w, v0.x, o[i][0]); o[i][1] = fmaf(w, v0.y, o[i][1]);
                        o[i][2] = fmaf(w, v0.z, o[i][2]); o[i][3] = fmaf(w, v0.w, o[i][3]);
                        if (DG == 2 && act1) {
                            o[i][4 * DG - 4] = fmaf(w, v1.x, o[i][4 * DG - 4]); o[i][4 * DG - 3] = fmaf(w, v1.y, o[i][4 * DG - 3]);
                            o[i][4 * DG - 2] = fmaf(w, v1.z, o[i][4 * DG - 2]); o[i][4 * DG - 1] = fmaf(w, v1.w, o[i][4 * DG - 1]);
                        }
                    }
                }
            }
            if (!whole) {
                const int jend = min(maxlim + 1, C::KW);
                int lim[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) lim[i] = row + 2 * i >= n ? -1 : min(masked ? row + 2 * i : n - 1, n - 1) - k0;
#pragma unroll 1
                for (int j = jfull; j < jend; ++j, ++pj, vj += C::DP) {
                    const float4 v0 = *reinterpret_cast<const float4*>(vj);
                    float4 v1 = v0;
                    if (DG == 2 && act1) v1 = *reinterpret_cast<const float4*>(vj + 64);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        if (j > lim[i]) continue;
                        const float w = pj[2 * i * C::PP];
                        o[i][0] = fmaf(w, v0.x, o[i][0]); o[i][1] = fmaf(w, v0.y, o[i][1]);
                        o[i][2] = fmaf(w, v0.z, o[i][2]); o[i][3] = fmaf(w, v0.w, o[i][3]);
                        if (DG == 2 && act1) {
                            o[i][4 * DG - 4] = fmaf(w, v1.x, o[i][4 * DG - 4]); o[i][4 * DG - 3] = fmaf(w, v1.y, o[i][4 * DG - 3]);
                            o[i][4 * DG - 2] = fmaf(w, v1.z, o[i][4 * DG - 2]); o[i][4 * DG - 1] = fmaf(w, v1.w, o[i][4 * DG - 1]);
                        }
                    }
                }
            }
        }
    }
    // ---- row sums over the 16 lanes of a row, the division of Eq. 2, output
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int off = 8; off; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
    if (KS == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (row + 2 * i >= n) continue;
            const float inv = 1.f / l[i];
            float* dst = out + base + (size_t)(row + 2 * i) * ld + 4 * tx;
#pragma unroll
            for (int g = 0; g < DG; ++g)
                if (g == 0 ? act0 : act1)
                    *reinterpret_cast<float4*>(dst + 64 * g) = make_float4(o[i][4 * g] * inv, o[i][4 * g + 1] * inv, o[i][4 * g + 2] * inv, o[i][4 * g + 3] * inv);
        }
    } else {
        // the KS partial results of a row, brought to their common maximum and added up
        __syncthreads();            // every warp is done with V and P
        float* part = Ks;           // [KS][BR][DP], over the K tile
        float* part_ml = Ps;        // [KS][BR] maxima, then [KS][BR] sums
        const int ks = warp % KS;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = qrow + 2 * i;
#pragma unroll
            for (int g = 0; g < DG; ++g)
                *reinterpret_cast<float4*>(part + (size_t)(ks * C::BR + r) * C::DP + 64 * g + 4 * tx) = make_float4(o[i][4 * g], o[i][4 * g + 1], o[i][4 * g + 2], o[i][4 * g + 3]);
            if (tx == 0) { part_ml[ks * C::BR + r] = m[i]; part_ml[KS * C::BR + ks * C::BR + r] = l[i]; }
        }
        __syncthreads();
        for (int t = tid; t < C::BR * d4; t += FA_THREADS) {
            const int r = t / d4, c = t - r * d4;
            if (r0 + r >= n) continue;
            float mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < KS; ++k) mx = fmaxf(mx, part_ml[k * C::BR + r]);
            float sum = 0.f;
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                const float mk = part_ml[k * C::BR + r];
                if (mk == -INFINITY && part_ml[KS * C::BR + k * C::BR + r] == 0.f) continue;      // no key of this share counts
                const float w = mk == mx ? 1.f : expf(mk - mx);
                const float4 f = *reinterpret_cast<const float4*>(part + (size_t)(k * C::BR + r) * C::DP + 4 * c);
                sum = fmaf(w, part_ml[KS * C::BR + k * C::BR + r], sum);
                y.x = fmaf(w, f.x, y.x); y.y = fmaf(w, f.y, y.y); y.z = fmaf(w, f.z, y.z); y.w = fmaf(w, f.w, y.w);
            }
            const float inv = 1.f / sum;
            *reinterpret_cast<float4*>(out + base + (size_t)(r0 + r) * ld + 4 * c) = make_float4(y.x * inv, y.y * inv, y.z * inv, y.w * inv);
        }
    }
    // ---- census
    for (int off = 16; off; off >>= 1) {
        dots += __shfl_xor_sync(0xffffffffu, dots, off);
        wts += __shfl_xor_sync(0xffffffffu, wts, off);
    }
    if (lane == 0) {
        if (MODE != 2 && dots) atomicAdd(&dc->qk_macs, (unsigned long long)dots * d);
        if (wts) { atomicAdd(&dc->pv_macs, (unsigned long long)wts * d); atomicAdd(&dc->exps, (unsigned long long)wts); }
    }
}

// ---------------------------------------------------------------- diagonal tiles of the masked scheme
// The weights inside a 128-row tile, j <= i, for the calls whose other blocks are on the tensor cores (f32_attn_tensor_kernel): maximum,
// sum and undivided output of every row, or the output itself where the tile is the head's first and so has nothing else.  A CTA per
// tile, all of it in shared memory.
//
// Phase 1 gives a thread 8 rows by 4 keys: 240 such pieces lie below the diagonal, one per thread of warps 0-7, and the 32 on it are
// warp 8's, which alone tests weight by weight.  Phase 3 gives a warp two groups of 8 rows, r and 15 - r, which together have 17 groups of
// 8 keys; the last group's triangle is unrolled.  Bound by the port of shared memory (12 loads of 16 bytes for 128 multiply-accumulates).
// Rows of Q and K are stored so that rows read at the same time are neighbours, 4 banks apart.
// Measured: the 128 tiles of 16 heads of n = 1024, d = 128 54 us as blocks of f32_flash_kernel, 30 here.
constexpr int FD_THREADS = 288, FD_CHAIN = 16;
template <int DG>
struct FDCfg {
    static constexpr int P = 64 * DG + 4, PP = 132;                      // row pitches of Q and K, of the weights, in floats
    static constexpr int QK = 128 * P, W = 128 * PP, V = 128 * 64 * DG;
    static constexpr int FRONT = 2 * QK > W ? 2 * QK : W;                // Q and K, then the weights over them
    static constexpr int SMEM = (FRONT + V + 256) * (int)sizeof(float);
};

template <int DG>
__global__ void __launch_bounds__(FD_THREADS, 3 - DG)
f32_diagonal_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V, float* __restrict__ out, float* __restrict__ ml,
                    const int* __restrict__ bad, int mark, int heads, int n, int H, int d, float scale, DeviceCounters* dc) {
    using C = FDCfg<DG>;
    extern __shared__ float4 fd_smem4[];
    float* Qs = reinterpret_cast<float*>(fd_smem4);
    float* Ks = Qs + C::QK;
    float* Ws = Qs;
    float* Vs = Qs + C::FRONT;
    float* row_m = Vs + C::V;
    float* row_l = row_m + 128;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bh = blockIdx.x % heads, tile = blockIdx.x / heads, b = bh / H, h = bh - b * H;
    grid_dependency_wait();
    if (bad[bh] == mark) return;
    const size_t ld = (size_t)H * d, base = ((size_t)b * n + tile * 128) * ld + (size_t)h * d;
    const int rows = min(128, n - tile * 128), d4 = d >> 2;
    for (int t = tid; t < 128 * d4; t += FD_THREADS) {
        const int r = t / d4, c = t - r * d4;
        if (r >= rows) continue;
        cp_async16(Qs + ((r & 7) * 16 + (r >> 3)) * C::P + 4 * c, Q + base + r * ld + 4 * c);       // row 8 r + i at 16 i + r
        cp_async16(Ks + ((r & 3) * 32 + (r >> 2)) * C::P + 4 * c, K + base + r * ld + 4 * c);       // row 4 c + u at 32 u + c
    }
    cp_async_commit();
    for (int t = tid; t < 128 * d4; t += FD_THREADS) {
        const int r = t / d4, c = t - r * d4;
        if (r < rows) cp_async16(Vs + r * 64 * DG + 4 * c, V + base + r * ld + 4 * c);
    }
    cp_async_commit();
    // zeros below the last row: nothing that is not a number may come in there
    for (int t = tid; t < (128 - rows) * d4; t += FD_THREADS) {
        const int r = rows + t / d4, c = t % d4;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(Qs + ((r & 7) * 16 + (r >> 3)) * C::P + 4 * c) = zero;
        *reinterpret_cast<float4*>(Ks + ((r & 3) * 32 + (r >> 2)) * C::P + 4 * c) = zero;
        *reinterpret_cast<float4*>(Vs + r * 64 * DG + 4 * c) = zero;
    }
    cp_async_wait_group<1>();
    __syncthreads();
    // ---- phase 1 (Eq. 1): piece (r, c) = rows 8 r .. 8 r + 7, keys 4 c .. 4 c + 3
    int r, c;
    if (warp < 8) {
        r = (int)((1.f + sqrtf(1.f + 4.f * tid)) * 0.5f);               // r (r - 1) <= tid < r (r + 1)
        if (r * (r - 1) > tid) --r;
        if (r * (r + 1) <= tid) ++r;
        c = tid - r * (r - 1);
    } else {
        r = lane >> 1;
        c = 2 * r + (lane & 1);
    }
    const bool have = warp == 8 || tid < 240;
    unsigned long long acc[8][4] = {};
    if (have) {
        const float* q = Qs + r * C::P;
        const float* k = Ks + c * C::P;
        auto step = [&](int x, auto edge_tag) {
            constexpr bool EDGE = decltype(edge_tag)::value;
            ulonglong2 kv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) kv[u] = *reinterpret_cast<const ulonglong2*>(k + 32 * u * C::P + 4 * x);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(q + 16 * i * C::P + 4 * x);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (!EDGE || 4 * (lane & 1) + u <= i) { fma2(acc[i][u], qv.x, kv[u].x); fma2(acc[i][u], qv.y, kv[u].y); }
            }
        };
        if (warp < 8) {
#pragma unroll 2
            for (int x = 0; x < d4; ++x) step(x, std::false_type{});
        } else {
#pragma unroll 1
            for (int x = 0; x < d4; ++x) step(x, std::true_type{});
        }
    }
    __syncthreads();                // every thread is done with Q and K
    if (have) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 f = unpack2(acc[i][u]);
                s[u] = (f.x + f.y) * scale;
            }
            *reinterpret_cast<float4*>(Ws + (8 * r + i) * C::PP + 4 * c) = make_float4(s[0], s[1], s[2], s[3]);
        }
    }
    cp_async_wait_all();
    __syncthreads();
    // ---- phase 2 (Eq. 2): two threads a row, alternating groups of four keys
    if (tid < 256) {
        const int row = tid >> 1, part = tid & 1;
        float* w = Ws + row * C::PP;
        float m = -INFINITY;
        for (int j = 4 * part; j <= row; j += 8) {
            const float4 f = *reinterpret_cast<const float4*>(w + j);
            m = fmaxf(m, f.x);
            if (j + 1 <= row) m = fmaxf(m, f.y);
            if (j + 2 <= row) m = fmaxf(m, f.z);
            if (j + 3 <= row) m = fmaxf(m, f.w);
        }
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        float s[4] = {0.f, 0.f, 0.f, 0.f};                              // (chains of 16)
        for (int j = 4 * part; j <= row; j += 8) {
            float4 f = *reinterpret_cast<const float4*>(w + j);
            f.x = expf(f.x - m); s[0] += f.x;
            if (j + 1 <= row) { f.y = expf(f.y - m); s[1] += f.y; }
            if (j + 2 <= row) { f.z = expf(f.z - m); s[2] += f.z; }
            if (j + 3 <= row) { f.w = expf(f.w - m); s[3] += f.w; }
            *reinterpret_cast<float4*>(w + j) = f;
        }
        float l = (s[0] + s[1]) + (s[2] + s[3]);
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        if (part == 0) {
            row_m[row] = m;
            row_l[row] = l;
            if (tile > 0 && row < rows) {
                ml[(size_t)bh * n + tile * 128 + row] = m;
                ml[((size_t)heads + bh) * n + tile * 128 + row] = l;
            }
        }
    }
    __syncthreads();
    // ---- phase 3 (Eq. 3): a lane has 2 DG columns of 8 rows
    constexpr int CW = 2 * DG;
    if (warp < 8 && CW * lane < d) {
        const float* v = Vs + CW * lane;
        auto value = [&](int j, float (&f)[CW]) {
            if constexpr (CW == 4) {
                const float4 t = *reinterpret_cast<const float4*>(v + j * 64 * DG);
                f[0] = t.x; f[1] = t.y; f[2] = t.z; f[3] = t.w;
            } else {
                const float2 t = *reinterpret_cast<const float2*>(v + j * 64 * DG);
                f[0] = t.x; f[1] = t.y;
            }
        };
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            const int g = side ? 15 - warp : warp;
            float o[8][CW] = {};
            const float* w = Ws + 8 * g * C::PP;
            // 16 keys at a time, then added up: with a chain over all of them the call had more error than f32_flash_kernel, whose chains are
            // split over warps (values of one sign, n = 385, d = 128 1.19e-7 and 0.89e-7 there, now 0.91e-7; 1-3 % of the call's time)
#pragma unroll 1
            for (int j0 = 0; j0 < 8 * g; j0 += FD_CHAIN) {
                float t[8][CW] = {};
#pragma unroll 1
                for (int j = j0; j < min(j0 + FD_CHAIN, 8 * g); j += 4) {
                    float4 p[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) p[i] = *reinterpret_cast<const float4*>(w + i * C::PP + j);
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        float f[CW];
                        value(j + jj, f);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float x = jj == 0 ? p[i].x : jj == 1 ? p[i].y : jj == 2 ? p[i].z : p[i].w;
#pragma unroll
                            for (int e = 0; e < CW; ++e) t[i][e] = fmaf(x, f[e], t[i][e]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int e = 0; e < CW; ++e) o[i][e] += t[i][e];
            }
            float t[8][CW] = {};
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {                    // the diagonal: rows from jj on
                float f[CW];
                value(8 * g + jj, f);
#pragma unroll
                for (int i = jj; i < 8; ++i) {
                    const float x = w[i * C::PP + 8 * g + jj];
#pragma unroll
                    for (int e = 0; e < CW; ++e) t[i][e] = fmaf(x, f[e], t[i][e]);
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int e = 0; e < CW; ++e) o[i][e] += t[i][e];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int row = 8 * g + i;
                if (row >= rows) continue;
                const float f = tile > 0 ? 1.f : 1.f / row_l[row];
                float* y = out + base + (size_t)row * ld + CW * lane;
                if constexpr (CW == 4) *reinterpret_cast<float4*>(y) = make_float4(o[i][0] * f, o[i][1] * f, o[i][2] * f, o[i][3] * f);
                else *reinterpret_cast<float2*>(y) = make_float2(o[i][0] * f, o[i][1] * f);
            }
        }
    }
    if (tid == 0) {
        const unsigned long long pairs = (unsigned long long)rows * (rows + 1) / 2;
        atomicAdd(&dc->qk_macs, pairs * d);
        atomicAdd(&dc->pv_macs, pairs * d);
        atomicAdd(&dc->exps, pairs);
    }
}

// Phase 1 of the symmetric scheme, tiled: one CTA per 64 x 64 block at or below the diagonal; S_ij for j <= i is computed
// once and stored at (i, j) and, through shared memory, at its mirror (j, i).
template <int DG>
__global__ void __launch_bounds__(FA_THREADS)
f32_sym_scores_kernel(const float* __restrict__ X, float* __restrict__ S, int n, int H, int d, float scale, DeviceCounters* dc) {
    using C = FACfg<DG, 1>;
    extern __shared__ float4 fa_smem4[];
    float* Qs = reinterpret_cast<float*>(fa_smem4);
    float* Ks = Qs + C::Q_FLOATS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tx = lane & 15, ty = lane >> 4;
    const int bh = blockIdx.x, b = bh / H, h = bh - b * H;
    int I = 0, t = blockIdx.y;
    while (t > I) { t -= I + 1; ++I; }
    const int r0 = 64 * I, c0 = 64 * t;
    const size_t ld = (size_t)H * d, base = ((size_t)b * n) * ld + (size_t)h * d;
    fa_load<DG, 64, C::DP, true>(Qs, X + base, r0, n, ld, d >> 2);
    fa_load<DG, 64, C::KP, false>(Ks, X + base, c0, n, ld, d >> 2);
    cp_async_wait_all();
    __syncthreads();
    const int qrow = 16 * warp + ty, row = r0 + qrow, wr0 = r0 + 16 * warp;
    int lim[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) lim[i] = row + 2 * i >= n ? -1 : row + 2 * i - c0;
    const int maxlim = wr0 >= n ? -1 : min(wr0 + 15, n - 1) - c0, minlim = wr0 + 15 >= n ? -1 : wr0 - c0;
    unsigned long long acc[8][4] = {}, dots = 0;
    if (minlim >= 63) fa_scores<DG, 4, false>(acc, Qs + qrow * C::DP, Ks + tx * C::KP, d >> 2, tx, ty, lim, minlim, maxlim);
    else if (maxlim >= 0) fa_scores<DG, 4, true>(acc, Qs + qrow * C::DP, Ks + tx * C::KP, d >> 2, tx, ty, lim, minlim, maxlim);
    __syncthreads();                // the operand tiles become the block's staging buffer, [64][65]
    float* Sh = S + (size_t)bh * n * n;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float2 f = unpack2(acc[i][u]);
            const float v = (f.x + f.y) * scale;
            const int j = tx + 16 * u;
            if (j > lim[i]) continue;
            Qs[(qrow + 2 * i) * 65 + j] = v;
            Sh[(size_t)(row + 2 * i) * n + c0 + j] = v;
            ++dots;
        }
    __syncthreads();
    for (int e = tid; e < 64 * 64; e += FA_THREADS) {       // mirror: row c0 + j, columns r0 + i
        const int j = e >> 6, i = e & 63;
        if (r0 + i < n && c0 + j < r0 + i) Sh[(size_t)(c0 + j) * n + r0 + i] = Qs[i * 65 + j];
    }
    for (int off = 16; off; off >>= 1) dots += __shfl_xor_sync(0xffffffffu, dots, off);
    if (lane == 0 && dots) atomicAdd(&dc->qk_macs, dots * (unsigned long long)d);
}

constexpr int ROWS_PER_BLOCK = 4;  // one warp per query row
constexpr int KEY_TILE = 32;

// MODE 0: all three phases for FULL / MASKED.
// MODE 1: phase 1 of the symmetric scheme: S_ij for j <= i, stored at (i,j) and at its mirror (j,i)
//         (the reuse of paper Sec. 4.1: the mirror costs a store, no MACs).
// MODE 2: phases 2 and 3 reading the weights' pre-softmax values from S.
template <int MODE>
__global__ void __launch_bounds__(ROWS_PER_BLOCK * 32)
f32_attn_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V,
                float* __restrict__ out, float* __restrict__ S, int n, int H, int d, float scale, int masked,
                DeviceCounters* dc, DeviceCounters* dc_next) {
    if (dc_next && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) *dc_next = DeviceCounters{0, 0, 0, 0, 0, 0, 0};      // (for the next call)
    extern __shared__ float sm[];
    float* ks = sm;                                   // [KEY_TILE][d + 1]
    float* qs = ks + KEY_TILE * (d + 1);              // [ROWS_PER_BLOCK][d]
    float* sc = qs + ROWS_PER_BLOCK * d;              // [ROWS_PER_BLOCK][n]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.z, h = blockIdx.y;
    const int i = blockIdx.x * ROWS_PER_BLOCK + warp;
    const bool live = i < n;
    const size_t ld = (size_t)H * d;                                  // row pitch of Q, K, V, out
    const size_t base = ((size_t)b * n) * ld + (size_t)h * d;
    const bool lower = (MODE == 1) || masked;                          // only j <= i is needed
    const int jend = live ? (lower ? i + 1 : n) : 0;                   // this warp's keys: [0, jend)
    const int last_row = min(n - 1, (int)blockIdx.x * ROWS_PER_BLOCK + ROWS_PER_BLOCK - 1);
    const int jend_block = lower ? last_row + 1 : n;
    float* myS = S ? S + ((size_t)(b * H + h) * n) * n : nullptr;
    float* mysc = sc + warp * n;
    unsigned long long dots = 0;

    if (MODE != 2) {
        if (live)
            for (int c = lane; c < d; c += 32) qs[warp * d + c] = Q[base + (size_t)i * ld + c];
        for (int j0 = 0; j0 < jend_block; j0 += KEY_TILE) {
            __syncthreads();
            for (int t = threadIdx.x; t < KEY_TILE * d; t += blockDim.x) {
                const int jj = t / d, c = t - jj * d;
                ks[jj * (d + 1) + c] = (j0 + jj < n) ? K[base + (size_t)(j0 + jj) * ld + c] : 0.f;
            }
            __syncthreads();
            const int j = j0 + lane;
            if (j < jend) {                                            // phase 1, Eq. 1: one weight per lane
                float acc = 0.f;
                const float* kr = ks + lane * (d + 1);
                const float* qr = qs + warp * d;
                for (int c = 0; c < d; ++c) acc = fmaf(qr[c], kr[c], acc);
                acc *= scale;
                ++dots;
                if (MODE == 1) {
                    myS[(size_t)i * n + j] = acc;
                    myS[(size_t)j * n + i] = acc;
                } else {
                    mysc[j] = acc;
                }
            }
        }
    } else {
        for (int j = lane; j < jend; j += 32) mysc[j] = myS[(size_t)i * n + j];
    }
    for (int off = 16; off; off >>= 1) dots += __shfl_xor_sync(0xffffffffu, dots, off);
    if (MODE != 2 && lane == 0 && dots) atomicAdd(&dc->qk_macs, dots * (unsigned long long)d);
    if (MODE == 1 || !live) return;
    __syncwarp();

    // phase 2, Eq. 2: exponent-accumulate over the kept weights, then normalisation
    float mx = -INFINITY;
    for (int j = lane; j < jend; j += 32) mx = fmaxf(mx, mysc[j]);
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    float sum = 0.f;
    for (int j = lane; j < jend; j += 32) {
        const float e = expf(mysc[j] - mx);
        mysc[j] = e;
        sum += e;
    }
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    __syncwarp();
    const float inv = 1.f / sum;

    // phase 3, Eq. 3: lanes own output components, keys are walked in order
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int j = 0; j < jend; ++j) {
        const float w = mysc[j];
        const float* vr = V + base + (size_t)j * ld;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int c = lane + 32 * t;
            if (c < d) acc[t] = fmaf(w, vr[c], acc[t]);
        }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int c = lane + 32 * t;
        if (c < d) out[base + (size_t)i * ld + c] = acc[t] * inv;
    }
    if (lane == 0) {
        atomicAdd(&dc->pv_macs, (unsigned long long)jend * d);
        atomicAdd(&dc->exps, (unsigned long long)jend);
    }
}

// ---------------------------------------------------------------- one launch for small layers
// Projections and the three phases of one (batch, head) in one CTA, everything in shared memory: the layer of a few
// dozen vectors is a few microseconds of work, and two launches with a round trip of q, k, v through global memory
// cost more than the arithmetic.  Element-exact skipping as in the kernels above: a weight the scheme does not need
// is never computed, and the census counts the multiply-accumulates actually executed.
constexpr int FS_THREADS = 512;
constexpr int FS_MAX_FLOATS = 56 * 1024;          // shared-memory budget in floats (224 KB)

struct FusedLayout {
    int xs_ld, t_ld, ds, s_ld;                    // row pitches: X, transposed q and k, v, the weight matrix S
    size_t xs, ws, qt, kt, vs, sm, rinv, total;   // offsets in floats
};
// q and k are kept transposed ([component][vector]) so that phase 1 reads four consecutive vectors of one component
// as one 16-byte access; v is kept [vector][component] for phase 3.
__host__ __device__ inline FusedLayout fused_layout(int n, int D, int d, int nW) {
    FusedLayout L;
    L.xs_ld = D + 1; L.t_ld = ((n + 3) & ~3) + 4; L.ds = d + 4; L.s_ld = n + 1;
    size_t off = 0;
    L.xs = off; off += (size_t)n * L.xs_ld; off = (off + 3) & ~size_t(3);
    L.ws = off; off += (size_t)nW * D * d;
    L.qt = off; off += (size_t)d * L.t_ld;
    L.kt = nW == 3 ? off : L.qt; if (nW == 3) off += (size_t)d * L.t_ld;
    L.vs = off; off += (size_t)n * L.ds;
    L.sm = off; off += (size_t)n * L.s_ld;
    L.rinv = off; off += n;
    L.total = off;
    return L;
}

__global__ void __launch_bounds__(FS_THREADS, 1)
f32_fused_layer_kernel(const float* __restrict__ X, const float* __restrict__ Wq, const float* __restrict__ Wk,
                       const float* __restrict__ Wv, float* __restrict__ out, int n, int H, int D, int d, float scale,
                       int scheme, DeviceCounters* dc, DeviceCounters* dc_next) {
    extern __shared__ float4 fs_smem4[];
    float* sm = reinterpret_cast<float*>(fs_smem4);
    grid_launch_dependents();     // (the next kernel may come in at once: its launch is hidden behind this one, its work is not)
    grid_dependency_wait();
    // the counter block of the NEXT call on this workspace is cleared here, off that call's critical path
    if (blockIdx.x == 0 && threadIdx.x == 0 && dc_next) *dc_next = DeviceCounters{0, 0, 0, 0, 0, 0, 0};
    const int nW = scheme == PSA_SYMMETRIC ? 1 : 3;
    const FusedLayout L = fused_layout(n, D, d, nW);
    float* xs = sm + L.xs; float* ws = sm + L.ws; float* qt = sm + L.qt; float* kt = sm + L.kt; float* vs = sm + L.vs;
    float* S = sm + L.sm; float* rinv = sm + L.rinv;
    const int b = blockIdx.x / H, h = blockIdx.x - b * H;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool lower = scheme != PSA_FULL;            // only j <= i is computed in phase 1 (masked; symmetric: then mirrored)
    const bool masked = scheme == PSA_MASKED;
    const size_t HD = (size_t)H * d;
    unsigned long long qk = 0, pv = 0, ex = 0;

    // ---- stage X[b] and this head's columns of the projection matrices (loads batched eight deep: a layer this small
    // lives on the latency of its first loads)
    {
        const float* xb = X + (size_t)b * n * D;
        for (int t0 = tid; t0 < n * D; t0 += 8 * FS_THREADS) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) { const int t = t0 + u * FS_THREADS; v[u] = t < n * D ? __ldg(xb + t) : 0.f; }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t0 + u * FS_THREADS;
                if (t < n * D) { const int i = t / D; xs[i * L.xs_ld + (t - i * D)] = v[u]; }
            }
        }
        const int d4 = d / 4;
        for (int w = 0; w < nW; ++w) {
            const float* W = (w == 0 ? Wq : (w == 1 ? Wk : Wv)) + (size_t)h * d;
            float4* dst = reinterpret_cast<float4*>(ws + (size_t)w * D * d);
            for (int t0 = tid; t0 < D * d4; t0 += 4 * FS_THREADS) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int t = t0 + u * FS_THREADS;
                    if (t < D * d4) { const int k = t / d4; v[u] = __ldg(reinterpret_cast<const float4*>(W + (size_t)k * HD) + (t - k * d4)); }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) { const int t = t0 + u * FS_THREADS; if (t < D * d4) dst[t] = v[u]; }
            }
        }
    }
    __syncthreads();

    // ---- projections (Sec. 3.1): 4 x 4 register tiles of q, k, v
    const int tr = (n + 3) / 4, tc = d / 4;
    for (int t = tid; t < nW * tr * tc; t += FS_THREADS) {
        const int w = t / (tr * tc), rem = t - w * tr * tc;
        const int i0 = (rem / tc) * 4, c0 = (rem % tc) * 4;
        const float* wp = ws + (size_t)w * D * d + c0;
        float acc[4][4] = {};
        int row[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) row[r] = min(i0 + r, n - 1) * L.xs_ld;
        for (int k = 0; k < D; ++k) {
            const float4 wv = *reinterpret_cast<const float4*>(wp + (size_t)k * d);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float x = xs[row[r] + k];
                acc[r][0] = fmaf(x, wv.x, acc[r][0]); acc[r][1] = fmaf(x, wv.y, acc[r][1]);
                acc[r][2] = fmaf(x, wv.z, acc[r][2]); acc[r][3] = fmaf(x, wv.w, acc[r][3]);
            }
        }
        if (w < 2) {          // q, k: transposed (rows beyond n land in the pitch's padding and are never used)
            float* dst = w == 0 ? qt : kt;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<float4*>(dst + (size_t)(c0 + u) * L.t_ld + i0) = make_float4(acc[0][u], acc[1][u], acc[2][u], acc[3][u]);
        }
        if (w == 2 || nW == 1) {   // v (the symmetric scheme's single projection is q, k and v at once)
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (i0 + r < n) *reinterpret_cast<float4*>(vs + (size_t)(i0 + r) * L.ds + c0) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
        }
    }
    __syncthreads();

    // ---- phase 1 (Eq. 1): S_ij = scale q_i . k_j for the weights the scheme needs, in 4 x 4 register tiles
    const int tn = (n + 3) / 4;
    for (int t = tid; t < tn * tn; t += FS_THREADS) {
        const int i0 = (t / tn) * 4, j0 = (t % tn) * 4;
        if (lower && j0 > i0 + 3) continue;                       // wholly above the diagonal: never issued
        const bool inside = i0 + 3 < n && j0 + 3 < n;
        if (inside && !(lower && j0 == i0)) {
            // a whole tile: 16 weights
            float acc[4][4] = {};
            for (int c = 0; c < d; ++c) {
                const float4 q4 = *reinterpret_cast<const float4*>(qt + (size_t)c * L.t_ld + i0);
                const float4 k4 = *reinterpret_cast<const float4*>(kt + (size_t)c * L.t_ld + j0);
                const float qv[4] = {q4.x, q4.y, q4.z, q4.w}, kv[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[r][u] = fmaf(qv[r], kv[u], acc[r][u]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float v = acc[r][u] * scale;
                    S[(size_t)(i0 + r) * L.s_ld + j0 + u] = v;
                    if (scheme == PSA_SYMMETRIC) S[(size_t)(j0 + u) * L.s_ld + i0 + r] = v;   // reuse (Sec. 4.1): a store, no MACs
                }
            qk += 16ull * d;
        } else if (inside) {
            // the tile on the diagonal of a lower-triangle scheme: the 10 weights with j <= i, nothing above them
            float acc[4][4] = {};
            for (int c = 0; c < d; ++c) {
                const float4 q4 = *reinterpret_cast<const float4*>(qt + (size_t)c * L.t_ld + i0);
                const float4 k4 = *reinterpret_cast<const float4*>(kt + (size_t)c * L.t_ld + j0);
                const float qv[4] = {q4.x, q4.y, q4.z, q4.w}, kv[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int u = 0; u <= r; ++u) acc[r][u] = fmaf(qv[r], kv[u], acc[r][u]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int u = 0; u <= r; ++u) {
                    const float v = acc[r][u] * scale;
                    S[(size_t)(i0 + r) * L.s_ld + j0 + u] = v;
                    if (scheme == PSA_SYMMETRIC) S[(size_t)(j0 + u) * L.s_ld + i0 + r] = v;
                }
            qk += 10ull * d;
        } else {
            // a tile that the edge of the matrix crosses (n not a multiple of 4): weight by weight
            for (int r = 0; r < 4; ++r)
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + r, j = j0 + u;
                    if (i >= n || j >= n || (lower && j > i)) continue;
                    float acc = 0.f;
                    for (int c = 0; c < d; ++c) acc = fmaf(qt[(size_t)c * L.t_ld + i], kt[(size_t)c * L.t_ld + j], acc);
                    acc *= scale;
                    S[(size_t)i * L.s_ld + j] = acc;
                    if (scheme == PSA_SYMMETRIC) S[(size_t)j * L.s_ld + i] = acc;
                    qk += d;
                }
        }
    }
    __syncthreads();

    // ---- phase 2 (Eq. 2): one warp per row; the division is applied to the output row
    for (int i = warp; i < n; i += FS_THREADS / 32) {
        const int jend = masked ? i + 1 : n;
        float* row = S + (size_t)i * L.s_ld;
        float mx = -INFINITY;
        for (int j = lane; j < jend; j += 32) mx = fmaxf(mx, row[j]);
        for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        float sum = 0.f;
        for (int j = lane; j < jend; j += 32) {
            const float e = expf(row[j] - mx);
            row[j] = e;
            sum += e;
        }
        for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (lane == 0) { rinv[i] = 1.f / sum; ex += (unsigned long long)jend; }
    }
    __syncthreads();

    // ---- phase 3 (Eq. 3): y_i = sum_j w_ij v_j over the kept weights, four output components per thread
    for (int t = tid; t < n * tc; t += FS_THREADS) {
        const int i = t / tc, c0 = (t - i * tc) * 4;
        const int jend = masked ? i + 1 : n;
        const float* row = S + (size_t)i * L.s_ld;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j = 0; j < jend; ++j) {
            const float w = row[j];
            const float4 v = *reinterpret_cast<const float4*>(vs + (size_t)j * L.ds + c0);
            acc.x = fmaf(w, v.x, acc.x); acc.y = fmaf(w, v.y, acc.y); acc.z = fmaf(w, v.z, acc.z); acc.w = fmaf(w, v.w, acc.w);
        }
        const float r = rinv[i];
        *reinterpret_cast<float4*>(out + ((size_t)b * n + i) * HD + (size_t)h * d + c0) = make_float4(acc.x * r, acc.y * r, acc.z * r, acc.w * r);
        pv += 4ull * jend;
    }

    // ---- census
    for (int off = 16; off; off >>= 1) {
        qk += __shfl_xor_sync(0xffffffffu, qk, off);
        pv += __shfl_xor_sync(0xffffffffu, pv, off);
        ex += __shfl_xor_sync(0xffffffffu, ex, off);
    }
    if (lane == 0) {
        if (qk) atomicAdd(&dc->qk_macs, qk);
        if (pv) atomicAdd(&dc->pv_macs, pv);
        if (ex) atomicAdd(&dc->exps, ex);
    }
    if (tid == 0) atomicAdd(&dc->proj_macs, (unsigned long long)nW * n * D * d);
}

// The same layer spread over a cluster of C CTAs (FULL and MASKED): 4-row tiles are dealt to the CTAs in turn (tile ti
// belongs to CTA ti % C, which balances the masked scheme's growing rows), each CTA projects q, k, v of its own rows, writes k
// and v into the shared memory of every CTA of the cluster, and finishes phases 1-3 for its rows.  A layer of one head then
// occupies C SMs instead of one.  The census is element-exact as above.
//
// What bounds it: latency.  A call of one head of n = 64, d_model = d = 64 is eight phases of one or two thousand cycles between barriers
// (clock stamps: first loads 2200, projections 2700, k and v to the other CTAs 1200 and their barrier 1200 .. 2700, phases 1-3 2200, 1100, 1300,
// output 1100).  So a phase is spread over all warps, sums in parts, loops have several loads in flight and no branch inside (with one per
// step the projections took 4100, phase 1 3500), and k and v rows are pushed (fetched by the CTAs that need them they took two barriers of the
// cluster and a pass of 3100 .. 4600).  The layout comes from the host, indices are divided by multiplication.
// Measured (us a call, among calls with other inputs; before / now): 1 head of n = 64, d = 64 masked 12.9 / 8.3, FULL 11.2 / 8.4; 12 heads FULL 11.8 / 8.6, 20 heads 22.6 / 10.9.
// Error against 64 bits (relative, 2-norm, 120 layers): 0.65 of that with undivided sums, nowhere more than 1 % larger.
struct ClusterLayout {
    int ld, s_ld;                            // row pitches: q, k, v; weights, kept as [key][own row]
    int tiles, group;                        // row tiles of a CTA (at most), rows that a task of the projections takes
    int keys;                                // keys that a warp takes in phase 1
    int splits, y_splits;                    // parts that a sum over components, over keys is taken in
    int xs, ws, part, qs, ks, vs, sm, rinv, y;
    size_t total;
    FastDiv by_columns, by_columns4, by_d, by_d4, by_key_groups, by_blocks;    // 3 d, 3 d / 4, d, d / 4, groups of keys, 32-column blocks
};
constexpr int FC_SPLITS = 8;
constexpr size_t FC_HALF_SM = 113 * 1024;     // shared memory of a CTA that leaves room for a second one
constexpr size_t FC_ALONE = FC_HALF_SM + 2048;     // that leaves none
inline ClusterLayout cluster_layout(int n, int D, int d, int C) {
    ClusterLayout L;
    L.tiles = ((n + 3) / 4 + C - 1) / C;
    L.group = L.tiles == 1 ? 4 : 8;
    L.ld = 4 * ((d / 4 + 1) | 1); L.s_ld = 4 * (L.tiles | 1);       // (odd numbers of 16 bytes: neighbouring rows lie in other banks)
    const int groups = (L.tiles + 1) / 2, rows = L.group * groups, blocks = L.tiles * ((d + 31) / 32), cols = 3 * d;
    L.keys = 8;                              // (four lanes to a key where one round of the warps does)
    while (L.keys < 32 && L.tiles * ((n + L.keys - 1) / L.keys) > FS_THREADS / 32) L.keys *= 2;
    L.y_splits = 1;
    while (2 * L.y_splits <= FC_SPLITS && 2 * L.y_splits * blocks <= FS_THREADS / 32) L.y_splits *= 2;
    L.xs = 0; L.ws = rows * D;
    L.sm = 0; L.rinv = n * L.s_ld; L.y = L.rinv + 4 * L.tiles;      // (these and q over x and W, once the projections are done)
    L.qs = L.y + L.y_splits * 4 * L.tiles * d;
    const int inputs = L.ws + cols * D, later = L.qs + rows * L.ld;
    L.ks = inputs > later ? inputs : later;
    L.vs = L.ks + n * L.ld;
    L.part = L.vs + n * L.ld;
    L.splits = 1;                            // (8 components each at least)
    while (2 * L.splits <= FC_SPLITS && 2 * L.splits * cols * groups <= FS_THREADS && 16 * L.splits <= D &&
           L.part + 2 * L.splits * rows * cols <= FS_MAX_FLOATS)
        L.splits *= 2;
    L.total = (size_t)L.part + L.splits * rows * cols;
    L.by_columns = fastdiv_make(cols); L.by_columns4 = fastdiv_make(cols / 4); L.by_d = fastdiv_make(d); L.by_d4 = fastdiv_make(d / 4);
    L.by_key_groups = fastdiv_make((n + L.keys - 1) / L.keys); L.by_blocks = fastdiv_make((d + 31) / 32);
    return L;
}

__global__ void __launch_bounds__(FS_THREADS, 2)
f32_fused_cluster_kernel(const float* __restrict__ X, const float* __restrict__ Wq, const float* __restrict__ Wk,
                         const float* __restrict__ Wv, float* __restrict__ out, int n, int H, int D, int d, float scale,
                         int scheme, DeviceCounters* dc, DeviceCounters* dc_next, const __grid_constant__ ClusterLayout L) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    extern __shared__ float4 fs_smem4[];
    float* sm = reinterpret_cast<float*>(fs_smem4);
    float* xs = sm + L.xs; float* ws = sm + L.ws; float* part = sm + L.part; float* qs = sm + L.qs; float* ks = sm + L.ks; float* vs = sm + L.vs;
    float* S = sm + L.sm; float* rinv = sm + L.rinv; float* ypart = sm + L.y;
    const int head = blockIdx.x / C, b = head / H, h = head - b * H;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int WARPS = FS_THREADS / 32;
    const bool masked = scheme == PSA_MASKED;
    const size_t HD = (size_t)H * d;
    const int tn = (n + 3) / 4;
    const int own_tiles = rank < tn ? (tn - rank + C - 1) / C : 0;     // tiles rank, rank + C, ...
    const int own_rows = 4 * own_tiles;                                // (rows beyond n, in the last tile only, are skipped)
    auto own_row = [&](int lr) { return 4 * (rank + (lr >> 2) * C) + (lr & 3); };     // local row -> row of the head
    const int valid_rows = own_tiles == 0 ? 0 : own_rows - max(0, own_row(own_rows - 1) + 1 - n);
    // The next kernel may come in at once: a call of one head takes 8 SMs, and the launch of the next one is hidden behind it.
    grid_launch_dependents();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // (every CTA has started: waited for ahead of the first remote store)
    grid_dependency_wait();
    if (blockIdx.x == 0 && tid == 0 && dc_next) *dc_next = DeviceCounters{0, 0, 0, 0, 0, 0, 0};

    // ---- stage this CTA's rows of X[b], as [group of rows][component][row], and the head's columns of the three projection matrices:
    // asynchronous copies, all in flight at once (a layer this small lives on the latency of its first loads)
    const int d4 = d / 4, gr = L.group, groups = (own_tiles + 1) / 2;
    {
        const float* xb = X + (size_t)b * n * D;
        for (int lr = warp; lr < gr * groups; lr += WARPS) {
            const int i = own_row(lr);
            const bool have = lr < valid_rows;
            float* dst = xs + (lr & -gr) * D + (lr & (gr - 1));
            for (int k = lane; k < D; k += 32) {
                if (have) cp_async4(dst + gr * k, xb + (size_t)i * D + k);
                else dst[gr * k] = 0.f;
            }
        }
        const int dk = fastdiv(FS_THREADS, L.by_d4), dc4 = FS_THREADS - dk * d4;
        int k = fastdiv(tid, L.by_d4), c4 = tid - k * d4;
        while (k < 3 * D) {
            const float* W = k < D ? Wq : k < 2 * D ? Wk - (size_t)D * HD : Wv - (size_t)2 * D * HD;
            cp_async16(ws + k * d + 4 * c4, W + (size_t)k * HD + (size_t)h * d + 4 * c4);
            k += dk; c4 += dc4;
            if (c4 >= d4) { c4 -= d4; ++k; }
        }
        cp_async_wait_all();
    }
    __syncthreads();

    // ---- projections (Sec. 3.1) of the own rows.  A task is one column of q, k or v for a group of rows and a part of the D components.
    const int splits = L.splits, step = (D + splits - 1) / splits, cols = 3 * d;
    for (int t = tid; t < cols * groups * splits; t += FS_THREADS) {
        const int rest = fastdiv(t, L.by_columns), col = t - rest * cols, g = rest >> __ffs(splits) - 1, p = rest & (splits - 1), which = fastdiv(col, L.by_d);
        const int k0 = p * step, k1 = min(D, k0 + step);
        const float* w = ws + (which * D + k0) * d + (col - which * d);
        float* dst = part + (p * groups + g) * gr * cols + col;
        auto rows = [&](auto rg_tag, const float* x) {
            constexpr int RG = decltype(rg_tag)::value;
            float acc[RG] = {};
#pragma unroll 8
            for (int k = k0; k < k1; ++k, w += d, x += RG) {
                const float wk = *w;
#pragma unroll
                for (int r = 0; r < RG; r += 4) {
                    const float4 f = *reinterpret_cast<const float4*>(x + r);
                    acc[r] = fmaf(f.x, wk, acc[r]); acc[r + 1] = fmaf(f.y, wk, acc[r + 1]);
                    acc[r + 2] = fmaf(f.z, wk, acc[r + 2]); acc[r + 3] = fmaf(f.w, wk, acc[r + 3]);
                }
            }
#pragma unroll
            for (int r = 0; r < RG; ++r) dst[r * cols] = acc[r];
        };
        if (gr == 4) rows(std::integral_constant<int, 4>{}, xs + 4 * (g * D + k0));
        else rows(std::integral_constant<int, 8>{}, xs + 8 * (g * D + k0));
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    // ---- the parts added up, four columns at a time: q stays here, k and v go to every CTA
    const int c4 = cols / 4;
    for (int t = tid; t < valid_rows * c4; t += FS_THREADS) {
        const int lr = fastdiv(t, L.by_columns4), q4 = t - lr * c4, i = own_row(lr);
        float4 s = *reinterpret_cast<const float4*>(part + lr * cols + 4 * q4);
        for (int p = 1; p < splits; ++p) {
            const float4 v = *reinterpret_cast<const float4*>(part + (p * groups * gr + lr) * cols + 4 * q4);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        const int which = fastdiv(q4, L.by_d4), c = 4 * (q4 - which * d4);
        if (which == 0) {
            *reinterpret_cast<float4*>(qs + lr * L.ld + c) = s;
        } else {
            float* dst = (which == 1 ? ks : vs) + i * L.ld + c;
            for (int r = 0; r < C; ++r) *reinterpret_cast<float4*>(cluster.map_shared_rank(dst, r)) = s;
        }
    }
    cluster.sync();           // every k and v row is here; no CTA reaches into another's shared memory from here on

    // ---- census of this CTA's rows: i + 1 (masked) or n weights each
    if (warp == 0) {
        unsigned pairs = 0;
        for (int lr = lane; lr < valid_rows; lr += 32) pairs += masked ? own_row(lr) + 1 : n;
        pairs = __reduce_add_sync(0xffffffffu, pairs);
        if (lane == 0 && pairs) {
            atomicAdd(&dc->qk_macs, (unsigned long long)pairs * d);
            atomicAdd(&dc->pv_macs, (unsigned long long)pairs * d);
            atomicAdd(&dc->exps, (unsigned long long)pairs);
            atomicAdd(&dc->proj_macs, (unsigned long long)valid_rows * cols * D);
        }
    }
    // ---- phase 1 (Eq. 1): S_ij = scale q_i . k_j.  A warp takes 32, 16 or 8 keys for the four rows of a tile; the lanes that share a key each
    // have every so-manieth group of four components.  A weight beyond the row's last kept key (masked: j > i; the edge) is never computed.
    const int keys = L.keys, lanes = 32 / keys, key_groups = (n + keys - 1) / keys;
    for (int unit = warp; unit < own_tiles * key_groups; unit += WARPS) {
        const int tile = fastdiv(unit, L.by_key_groups), j = keys * (unit - tile * key_groups) + (lane & (keys - 1)), p = lane / keys, i0 = own_row(4 * tile);
        const int first = masked ? max(0, j - i0) : 0, last = j < n ? min(4, n - i0) : 0;     // rows first .. last - 1 of the tile keep key j
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        if (first < last) {
            const float* k = ks + j * L.ld;
            const float* q = qs + 4 * tile * L.ld;
#pragma unroll 4
            for (int c = 4 * p; c < d; c += 4 * lanes) {
                const float4 kv = *reinterpret_cast<const float4*>(k + c);
                float4 qv[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) qv[r] = *reinterpret_cast<const float4*>(q + r * L.ld + c);
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (r >= first && r < last) {
                        acc[r] = fmaf(qv[r].x, kv.x, acc[r]); acc[r] = fmaf(qv[r].y, kv.y, acc[r]);
                        acc[r] = fmaf(qv[r].z, kv.z, acc[r]); acc[r] = fmaf(qv[r].w, kv.w, acc[r]);
                    }
            }
        }
        for (int off = keys; off < 32; off *= 2) {
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r >= first && r < last && (r & (lanes - 1)) == p) S[j * L.s_ld + 4 * tile + r] = acc[r] * scale;
    }
    __syncthreads();

    // ---- phase 2 (Eq. 2): one warp per own row; the division is applied to the output row
    for (int lr = warp; lr < valid_rows; lr += WARPS) {
        const int jend = masked ? own_row(lr) + 1 : n;
        float* row = S + lr;
        float mx = -INFINITY;
        for (int j = lane; j < jend; j += 32) mx = fmaxf(mx, row[j * L.s_ld]);
        for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        float sum = 0.f;
        for (int j = lane; j < jend; j += 32) {
            const float e = expf(row[j * L.s_ld] - mx);
            row[j * L.s_ld] = e;
            sum += e;
        }
        for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (lane == 0) rinv[lr] = 1.f / sum;
    }
    __syncthreads();

    // ---- phase 3 (Eq. 3): y_i = sum_j w_ij v_j over the kept weights.  A warp takes up to 32 columns of a tile's four rows; the keys are
    // split among y_splits warps, and among a warp's lanes where there are less than 32 columns.
    const int width = d <= 8 ? 8 : d <= 16 ? 16 : 32, blocks = (d + 31) / 32, ysplits = L.y_splits;
    for (int unit = warp; unit < own_tiles * blocks * ysplits; unit += WARPS) {
        const int rest = unit >> __ffs(ysplits) - 1, p = unit - rest * ysplits, tile = fastdiv(rest, L.by_blocks), c = 32 * (rest - tile * blocks) + (lane & (width - 1));
        // keys that all four rows keep, that any row keeps; neither goes beyond n, so that no v row beyond the sequence is read.  (Where n is no multiple
        // of 4, the last tile's rows beyond n have q and weights of whatever shared memory held before, here as in phase 1: each row has an
        // accumulator of its own, and those rows' are never stored.)
        const int i0 = own_row(4 * tile), whole = masked ? i0 + 1 : n, jend = masked ? min(i0 + 4, n) : n, step = ysplits * (32 / width);
        const float* w = S + 4 * tile;
        const float* v = vs + min(c, d - 1);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        int j = p + ysplits * (lane / width);
#pragma unroll 4
        for (; j < whole; j += step) {
            const float4 wj = *reinterpret_cast<const float4*>(w + j * L.s_ld);
            const float x = v[j * L.ld];
            acc[0] = fmaf(wj.x, x, acc[0]); acc[1] = fmaf(wj.y, x, acc[1]); acc[2] = fmaf(wj.z, x, acc[2]); acc[3] = fmaf(wj.w, x, acc[3]);
        }
#pragma unroll 1
        for (; j < jend; j += step) {
            const float x = v[j * L.ld];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (j <= i0 + r) acc[r] = fmaf(w[j * L.s_ld + r], x, acc[r]);
        }
        __syncwarp();
        for (int off = width; off < 32; off *= 2) {
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
        }
        if (lane < width && c < d) {
#pragma unroll
            for (int r = 0; r < 4; ++r) ypart[(p * own_rows + 4 * tile + r) * d + c] = acc[r];
        }
    }
    __syncthreads();
    for (int lr = warp / 2; lr < valid_rows; lr += WARPS / 2) {        // two warps a row
        float* y = out + ((size_t)b * n + own_row(lr)) * HD + (size_t)h * d;
        const float f = rinv[lr];
        for (int c = 32 * (warp & 1) + lane; c < d; c += 64) {
            float s = ypart[lr * d + c];
            for (int p = 1; p < ysplits; ++p) s += ypart[(p * own_rows + lr) * d + c];
            y[c] = s * f;
        }
    }
}

size_t attn_smem_bytes(int n, int d) {
    return sizeof(float) * ((size_t)KEY_TILE * (d + 1) + (size_t)ROWS_PER_BLOCK * d + (size_t)ROWS_PER_BLOCK * n);
}

}  // namespace

namespace {
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The general kernels count row tiles, or sequences, in a grid dimension that holds 65535: calls with more go in several launches.
constexpr int GRID_MAX = 65535;

cudaError_t project_general(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D, int N,
                            const float* residual, DeviceCounters* dc, cudaStream_t stream) {
    constexpr int SLICE = GRID_MAX * PROJ_TILE;
    for (int r0 = 0; r0 < rows; r0 += min(SLICE, rows - r0)) {
        const int nr = min(SLICE, rows - r0);
        const size_t o = (size_t)r0 * N;
        const dim3 block(PROJ_TILE, PROJ_TILE), grid((N + PROJ_TILE - 1) / PROJ_TILE, (nr + PROJ_TILE - 1) / PROJ_TILE, nW);
        f32_project_kernel<<<grid, block, 0, stream>>>(X + (size_t)r0 * D, W[0], W[1], W[2], out[0] + o, out[1] + o, out[2] + o, nr, D, N,
                                                       residual ? residual + o : nullptr, dc);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t attention_general(const float* Q, const float* K, const float* V, float* out, float* S, int B, int H, int n, int d,
                              float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next, cudaStream_t stream) {
    const size_t smem = attn_smem_bytes(n, d);
    for (int b0 = 0; b0 < B; b0 += min(GRID_MAX, B - b0)) {
        const int nb = min(GRID_MAX, B - b0);
        const size_t o = (size_t)b0 * n * H * d;
        const dim3 grid((n + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK, H, nb), block(ROWS_PER_BLOCK * 32);
        if (scheme == PSA_SYMMETRIC) {
            float* s = S + (size_t)b0 * H * n * n;
            f32_attn_kernel<1><<<grid, block, smem, stream>>>(Q + o, Q + o, Q + o, out + o, s, n, H, d, scale, 0, dc, nullptr);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            f32_attn_kernel<2><<<grid, block, smem, stream>>>(Q + o, Q + o, Q + o, out + o, s, n, H, d, scale, 0, dc, dc_next);
        } else {
            f32_attn_kernel<0><<<grid, block, smem, stream>>>(Q + o, K + o, V + o, out + o, nullptr, n, H, d, scale, scheme == PSA_MASKED ? 1 : 0, dc, dc_next);
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
}  // namespace

cudaError_t f32_project(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D,
                        int N, const float* residual, const F32ProjectScratch* ps, DeviceCounters* dc, cudaStream_t stream) {
    bool tiled = D % 4 == 0 && N % 4 == 0 && aligned16(X) && aligned16(residual);      // 16-byte rows
    for (int w = 0; w < nW; ++w) tiled = tiled && aligned16(W[w]) && aligned16(out[w]);
    if (tiled) {
        static DeviceSetup setup;
        const int sms = device_setup(&setup, [] { return cudaSuccess; }, "fp32 projection set-up");
        if (sms <= 0) return cudaErrorUnknown;
        // Bound by the latency of their k-steps, the smallest calls run best on the 16 x 16 tiles of the general kernel, as long
        // as these are not more than the SMs (by the library's events, us, 16 x 16 / 32 x 32: 96 x 768 x 3 x 64, 72 tiles, 22.8 /
        // 24.7; 16 x 768 x 3 x 768, 144 tiles, 22.9 / 24.9; 200 x 768 x 3 x 64, 156 tiles, 25.5 / 24.8; 128 x 2048 x 64, 32 tiles,
        // 51.2 / 55.0), for calls of one row of tiles up to three times that (16 x 1024 x 3 x 2048, 384 tiles, 43.2 / 46.6).
        const long long tiles16 = (long long)((rows + 15) / 16) * ((N + 15) / 16) * nW;
        if (tiles16 <= (rows <= 16 ? 3 * sms : sms)) return project_general(X, W, out, nW, rows, D, N, residual, dc, stream);
        // The tensor cores from two 32 x 32 tiles per SM on, by measurement (us, 32 x 32 tiles on CUDA cores / tensor cores):
        // 64 x 768 x 3 x 64 23.5 / 32.3, 128 x 768 x 3 x 768 (288 tiles) 29.6 / 33.6, 2048 x 768 x 3 x 64 (384) 37.5 / 33.4,
        // 600 x 320 x 3 x 320 (570) 27.3 / 21.3, 64 x 2048 x 3 x 2048 (384) 89 / 72; larger ones, against 128 x 128 tiles on CUDA
        // cores, 2048 x 768 x 3 x 768 171 / 70.
        const long long tiles = (long long)((rows + 31) / 32) * ((N + 31) / 32) * nW;
        if (ps && f32_project_pairs_fit(rows, D, N, nW, ps->bytes) && f32_project_pairs_pay(rows, D, N, nW, sms))
            return f32_project_pairs(X, W, out, nW, rows, D, N, residual, ps->parts, ps->marks, ps->mark, dc, stream);
        if (tiles > 2 * sms) return f32_project_tensor(X, W, out, nW, rows, D, N, residual, dc, stream);
        const dim3 grid((N + GP_BN - 1) / GP_BN, (rows + GP_BM - 1) / GP_BM, nW);
        f32_project_tiled_kernel<<<grid, GP_THREADS, GP_SMEM, stream>>>(X, W[0], W[1], W[2], out[0], out[1], out[2], rows, D, N, residual, dc);
        return cudaGetLastError();
    }
    return project_general(X, W, out, nW, rows, D, N, residual, dc, stream);
}

bool f32_fused_fits(int n, int D, int d, int scheme) {
    if (n > 256 || d % 4 != 0 || d > 128) return false;
    return fused_layout(n, D, d, scheme == PSA_SYMMETRIC ? 1 : 3).total <= (size_t)FS_MAX_FLOATS;
}

// Heads few enough that one CTA each would leave SMs idle are spread over clusters: of the largest size of which all clusters of the call fit the GPU at
// once, each CTA alone on its SM (by the shared memory that it asks for).  A cluster stays inside a part of the GPU, so that fewer fit than SMs / size; the
// runtime says how many, and steps lie where it says: 15 of 8, 33 of 4 and 74 of 2 on 148 SMs.  Masked, n = 64, d_model = d = 64, us for a CTA per head / clusters of
// 2 / 4 / 8 alone: 15 heads 24.6 15.2 10.5 8.5, 16 24.6 15.2 10.5 15.9, 33 24.6 15.4 10.5 23.9, 34 24.6 15.4 19.8 23.9, 74 24.6 15.3 29.7 40.2, 80 24.6 29.6 29.8.
// Clusters that share SMs pack while others are idle (12 heads 8.5 alone, 12.5 sharing), but 71 of 4 fit then, and up to 64 heads, a tenth of the GPU left free, take
// these before clusters of 2: 34 heads of n = 150, d = 16 18.1 against 19.4, 48 of n = 96, d = 48 20.6 against 20.9 (short heads lose, 48 of n = 64, d = 64 16.2 against
// 15.3, d = 16 10.2 against 9.5, but with half as many CTAs to a head sums are split less and the error against 64 bits grows by up to a fifth).
// Many heads of up to 16 vectors gain nothing (48 of n = 16, d = 16 8.0, clusters of 2 or 4 7.6).
struct ClusterFits {
    int alone[3], sharing4;                  // clusters of 2, 4, 8 CTAs alone on their SMs; of 4, two CTAs to an SM
};
ClusterFits g_cluster_fits[MAX_DEVICES];
cudaError_t clusters_that_fit(int c, size_t bytes, int* clusters) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(FS_THREADS);
    cfg.dynamicSmemBytes = bytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, f32_fused_cluster_kernel, &cfg);
}
cudaError_t fused_setup() {
    constexpr int bytes = FS_MAX_FLOATS * (int)sizeof(float);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f32_fused_layer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f32_fused_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    ClusterFits& f = g_cluster_fits[dev];
    for (int i = 0; i < 3 && e == cudaSuccess; ++i) e = clusters_that_fit(2 << i, FC_ALONE, &f.alone[i]);
    if (e == cudaSuccess) e = clusters_that_fit(4, FC_HALF_SM, &f.sharing4);
    return e;
}
int f32_fused_cluster_size(int B, int H, int n, int D, int d, int scheme, const ClusterFits& f, bool* alone) {
    const long long heads = (long long)B * H;
    *alone = true;
    if (scheme == PSA_SYMMETRIC || (heads > 32 && n <= 16)) return 1;      // (the symmetric scheme's mirrored store crosses row owners)
    auto bytes = [&](int c) { return cluster_layout(n, D, d, c).total * sizeof(float); };
    auto fits = [&](int c) { return c <= (n + 3) / 4 && bytes(c) <= FS_MAX_FLOATS * sizeof(float); };
    if (heads <= f.alone[2] && fits(8)) return 8;
    if (heads <= f.alone[1] && fits(4)) return 4;
    if (heads <= f.sharing4 - f.sharing4 / 10 && fits(4) && bytes(4) <= FC_HALF_SM) { *alone = false; return 4; }
    return heads <= f.alone[0] && fits(2) ? 2 : 1;
}

cudaError_t f32_fused_layer(const float* X, const float* Wq, const float* Wk, const float* Wv, float* out, int B, int H,
                            int n, int D, int d, float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next,
                            cudaStream_t stream) {
    static DeviceSetup setup;
    int dev = 0;
    if (device_setup(&setup, fused_setup, "fp32 fused layer set-up", &dev) <= 0) return cudaErrorUnknown;
    bool alone;
    const int C = f32_fused_cluster_size(B, H, n, D, d, scheme, g_cluster_fits[dev], &alone);
    if (C > 1) {
        const ClusterLayout L = cluster_layout(n, D, d, C);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(B * H * C);
        cfg.blockDim = dim3(FS_THREADS);
        cfg.dynamicSmemBytes = std::max(L.total * sizeof(float), alone ? FC_ALONE : 0);
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        return cudaLaunchKernelEx(&cfg, f32_fused_cluster_kernel, X, Wq, Wk, Wv, out, n, H, D, d, scale, scheme, dc, dc_next, L);
    }
    const size_t smem = fused_layout(n, D, d, scheme == PSA_SYMMETRIC ? 1 : 3).total * sizeof(float);
    f32_fused_layer_kernel<<<B * H, FS_THREADS, smem, stream>>>(X, Wq, scheme == PSA_SYMMETRIC ? Wq : Wk,
                                                               scheme == PSA_SYMMETRIC ? Wq : Wv, out, n, H, D, d, scale,
                                                               scheme, dc, dc_next);
    return cudaGetLastError();
}

namespace {
template <int DG, int KS, int MODE>
cudaError_t launch_flash(const float* Q, const float* K, const float* V, float* out, const float* S, int B, int H, int n, int d,
                         float scale, int masked, DeviceCounters* dc, DeviceCounters* dc_next, const F32Scratch* fs, cudaStream_t stream) {
    using C = FACfg<DG, KS>;
    static DeviceSetup setup;
    if (device_setup(&setup, [] {
            return cudaFuncSetAttribute(f32_flash_kernel<DG, KS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, FACfg<DG, KS>::SMEM);
        }, "fp32 attention set-up") <= 0)
        return cudaErrorUnknown;
    const dim3 grid(B * H, (n + C::BR - 1) / C::BR);
    if (!fs) {
        f32_flash_kernel<DG, KS, MODE><<<grid, FA_THREADS, C::SMEM, stream>>>(Q, K, V, out, S, n, H, d, scale, masked, dc, dc_next, nullptr, 0);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(FA_THREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // (waits for its predecessor itself)
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f32_flash_kernel<DG, KS, MODE>, Q, K, V, out, S, n, H, d, scale, masked, dc, dc_next, static_cast<const int*>(fs->bad), fs->mark);
}
template <int DG, int MODE>
cudaError_t launch_flash_split(const float* Q, const float* K, const float* V, float* out, const float* S, int B, int H, int n,
                               int d, float scale, int masked, DeviceCounters* dc, DeviceCounters* dc_next, const F32Scratch* fs, int sms, cudaStream_t stream) {
    auto ctas = [&](int br) { return (long long)B * H * ((n + br - 1) / br); };
    // Fewer rows per CTA cost efficiency (every warp rereads K for 16 rows, with 4 / KS keys to a load of q) and buy CTAs: the
    // line lies at two CTAs per SM (us for KS = 1 / 2 / 4).  16 heads of n = 300, d = 64, 80 tiles of 64 rows: 70 / 44 / 35; 16 of
    // n = 1024, d = 128, masked, 256 tiles: 210 / 166 / 216; 74 of n = 256, d = 64, 296 tiles: 46 / 54 / 70; 48 of n = 512, d = 64, 384
    // tiles: 110 / 124 / 159.  It is not exact: 16 heads of n = 1024, FULL, d = 64 161 / 179 / 208; 64 of n = 300, 320 tiles with a
    // nearly empty last one, 101 / 82 / 87.
    if (ctas(64) >= 2 * sms) return launch_flash<DG, 1, MODE>(Q, K, V, out, S, B, H, n, d, scale, masked, dc, dc_next, fs, stream);
    if (ctas(32) >= 2 * sms) return launch_flash<DG, 2, MODE>(Q, K, V, out, S, B, H, n, d, scale, masked, dc, dc_next, fs, stream);
    return launch_flash<DG, 4, MODE>(Q, K, V, out, S, B, H, n, d, scale, masked, dc, dc_next, fs, stream);
}
template <int DG>
cudaError_t tiled_attention(const float* Q, const float* K, const float* V, float* out, float* S, int B, int H, int n, int d,
                            float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next, int sms, cudaStream_t stream) {
    if (scheme != PSA_SYMMETRIC)
        return launch_flash_split<DG, 0>(Q, K, V, out, nullptr, B, H, n, d, scale, scheme == PSA_MASKED, dc, dc_next, nullptr, sms, stream);
    constexpr int SMEM = (FACfg<DG, 1>::Q_FLOATS + FACfg<DG, 1>::K_FLOATS) * (int)sizeof(float);
    static DeviceSetup setup;
    if (device_setup(&setup, [] {
            return cudaFuncSetAttribute(f32_sym_scores_kernel<DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
        }, "fp32 scores set-up") <= 0)
        return cudaErrorUnknown;
    const int T = (n + 63) / 64;
    f32_sym_scores_kernel<DG><<<dim3(B * H, T * (T + 1) / 2), FA_THREADS, SMEM, stream>>>(Q, S, n, H, d, scale, dc);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_flash_split<DG, 2>(Q, Q, Q, out, S, B, H, n, d, scale, 0, dc, dc_next, nullptr, sms, stream);
}
// The call on the tensor cores (psa_f32_attn_tensor.cu), with the weights on the diagonal tiles and the heads that path cannot take here.
template <int DG>
cudaError_t tensor_attention(const float* Q, const float* K, const float* V, float* out, const F32Scratch& fs, int B, int H, int n, int d, float scale,
                             int masked, DeviceCounters* dc, DeviceCounters* dc_next, int sms, cudaStream_t stream) {
    cudaError_t e = f32_attention_split(Q, K, V, fs, B, H, n, d, stream);
    if (e == cudaSuccess && masked) {
        static DeviceSetup setup;
        if (device_setup(&setup, [] {
                return cudaFuncSetAttribute(f32_diagonal_kernel<DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, FDCfg<DG>::SMEM);
            }, "fp32 diagonal tiles set-up") <= 0)
            return cudaErrorUnknown;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(B * H * ((n + 127) / 128));
        cfg.blockDim = dim3(FD_THREADS);
        cfg.dynamicSmemBytes = FDCfg<DG>::SMEM;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // (waits for its predecessor itself)
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, f32_diagonal_kernel<DG>, Q, K, V, out, fs.ml, static_cast<const int*>(fs.bad), fs.mark, B * H, n, H, d, scale, dc);
    }
    if (e == cudaSuccess) e = f32_attention_tensor(Q, out, fs, B, H, n, d, scale, masked, dc, stream);
    if (e == cudaSuccess) e = launch_flash_split<DG, 0>(Q, K, V, out, nullptr, B, H, n, d, scale, masked, dc, dc_next, &fs, sms, stream);
    return e;
}
}  // namespace

namespace {
// Whether the general kernel, a warp per row and many small CTAs per SM, is the faster one: heads of few vectors.  The tiled
// one has two or three CTAs per SM, in each of which one warp of four has work then, and the symmetric scheme's takes 64 x 64
// blocks whatever the length.  Measured on 148 SMs (us, general / tiled).  FULL; MASKED is alike up to d = 64: 1024 heads of n = 8,
// d = 16 22.7 / 26.5, n = 12 30.9 / 27.4; d = 64, n = 8 26.8 / 41.0, n = 12 36.0 / 42.5, n = 16 46.2 / 42.3; up to a head per SM no
// difference (148 heads of n = 12, d = 128: 16.6 / 14.5).  d > 64: 230 heads of n = 10, d = 128 16.6 / 12.6.  d = 68: 296 heads of n = 18
// 22.7 / 20.7, 400 heads 28.9 / 35.0, 1500 heads of n = 24 88 / 112; 512 heads, which fill two rounds of the tiled kernel better,
// of n = 16 30.9 / 29.0, of n = 28 47.7 / 45.6.  d = 128: 400 heads of n = 28
// 48.8 / 57.5, 1024 heads 103 / 115, 1180 heads 127 / 116, of n = 24 94 / 104, 1500 heads 129 / 154; 4096 heads of n = 16 253 / 269,
// n = 20 360 / 330.  MASKED, where the general kernel skips more: 4096 heads of n = 20, d = 68 196 / 234, d = 128 301 / 330, of n = 24
// 267 / 253, 398 / 350.  Symmetric: a head of n = 8, d = 16 14.3 / 14.5, d = 64 14.2 / 18.6, d = 128 14.4 / 28.8; 1024 heads of d = 16,
// n = 9 28.8 / 32.9, n = 12 35.1 / 32.9, 400 heads of n = 10 18.6 / 16.6; d = 64, n = 12 39.9 / 47.3, n = 16 51.8 / 47.3; d = 128, n = 20 84 / 92, n = 24 99 / 100, 400 heads
// of n = 14 33.5 / 39.1, n = 16 35.9 / 33.0, 150 heads of n = 28 30.5 / 37.4; 64 heads of n = 28, d = 32 16.6 / 16.6, n = 32, d = 64 18.6 / 19.1, n = 40, d = 128 33.0 / 32.9.
bool short_heads(long long heads, int n, int d, int scheme, int sms) {
    const bool masked = scheme == PSA_MASKED;
    if (scheme == PSA_SYMMETRIC) {
        if (n <= (d <= 16 ? (heads > 3 * sms ? 9 : 8) : 12)) return true;
        if (2 * heads <= sms) return d > 16 && n <= (d <= 64 ? 32 : 40);
        if (d <= 64 || n > (2 * heads <= 3 * sms ? 28 : 20)) return false;
        return n < 16 || heads > 3 * sms || (n == 16 ? 2 * heads <= 3 * sms : heads < 2 * sms);
    }
    if (heads <= sms || (d > 64 && heads < 2 * sms)) return false;
    if (n <= (d <= 16 ? 8 : d <= 48 ? 10 : 12)) return true;
    if (d <= 64 || heads <= 2 * sms) return false;
    if (d <= 80 && heads > 3 * sms && heads <= 4 * sms && (n > 20 || (n == 16 && !masked))) return false;
    return n <= (heads <= 7 * sms ? 28 : heads <= 11 * sms ? 24 : masked ? 20 : 16);
}
}  // namespace

cudaError_t f32_attention(const float* Q, const float* K, const float* V, float* out, float* S, const F32Scratch* fs, int B, int H,
                          int n, int d, float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next, cudaStream_t stream) {
    static DeviceSetup setup;
    const int sms = device_setup(&setup, [] { return cudaSuccess; }, "fp32 attention set-up");
    if (sms <= 0) return cudaErrorUnknown;
    if (fs && f32_tensor_attention_fits(B, H, n, d, scheme))
        return d <= 64 ? tensor_attention<1>(Q, K, V, out, *fs, B, H, n, d, scale, scheme == PSA_MASKED, dc, dc_next, sms, stream)
                       : tensor_attention<2>(Q, K, V, out, *fs, B, H, n, d, scale, scheme == PSA_MASKED, dc, dc_next, sms, stream);
    if (H <= GRID_MAX && short_heads((long long)B * H, n, d, scheme, sms))
        return attention_general(Q, K, V, out, S, B, H, n, d, scale, scheme, dc, dc_next, stream);
    if (d % 4 == 0 && (long long)B * H <= 0x7fffffff && aligned16(Q) && aligned16(K) && aligned16(V) && aligned16(out))      // 16-byte rows
        return d <= 64 ? tiled_attention<1>(Q, K, V, out, S, B, H, n, d, scale, scheme, dc, dc_next, sms, stream)
                       : tiled_attention<2>(Q, K, V, out, S, B, H, n, d, scale, scheme, dc, dc_next, sms, stream);
    return attention_general(Q, K, V, out, S, B, H, n, d, scale, scheme, dc, dc_next, stream);
}

}  // namespace psa
