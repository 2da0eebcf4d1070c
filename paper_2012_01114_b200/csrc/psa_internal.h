// Internal declarations shared by the translation units of libpsa (not part of the public interface).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/psa.h"

namespace psa {

// Device-resident counters of one call, zeroed (stream-ordered) before its first kernel.
// Kernels add to them once per block of work they actually issue.
struct DeviceCounters {
    unsigned long long proj_macs;
    unsigned long long qk_macs;
    unsigned long long pv_macs;
    unsigned long long exps;
    int status;  // PSA_OK or PSA_ERR_TIMEOUT
    unsigned int next_item;  // work-list cursor of the persistent attention kernel
    // (row, key block) events of the bf16 online softmax in which a row's running maximum was raised after the
    // row's first block, so that its partial output and row sum were rescaled (diagnostic, psa_last_rescales)
    unsigned long long rescales;
};

// ---- fp32 CUDA-core path (psa_f32.cu) ----
// out[w][r, c] = sum_k X[r, k] W[w][k, c] for w < nW.
// `residual` ([rows, N], may be null) is added to every output.
// `ps` (may be null): scratch for the largest calls, see f32_project_pairs; `bytes`: room for the parts; `mark`: what a mark of this call is (any other
// number is none, so that marks need not be clear when a call starts).
struct F32ProjectScratch {
    void* parts;
    size_t bytes;
    int* marks;
    int mark;
};
cudaError_t f32_project(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D,
                        int N, const float* residual, const F32ProjectScratch* ps, DeviceCounters* dc, cudaStream_t stream);
// The same on the tensor cores, to the same accuracy (psa_f32_tensor.cu); f32_project chooses.  Rows of 16 bytes, as there.
cudaError_t f32_project_tensor(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D, int N,
                               const float* residual, DeviceCounters* dc, cudaStream_t stream);
// The same for the largest calls, operands split once into `parts` (f32_project_parts_bytes, psa_ws.h), on pairs of CTAs.  marks:
// f32_project_marks ints, none of them `mark` when the call's kernels start.
bool f32_project_pairs_pay(int rows, int D, int N, int nW, int sms);
cudaError_t f32_project_pairs(const float* X, const float* const W[3], float* const out[3], int nW, int rows, int D, int N, const float* residual,
                              void* parts, int* marks, int mark, DeviceCounters* dc, cudaStream_t stream);
// Scratch of the tensor-core attention: marks of the heads it cannot take (B H ints, set to `mark`, which none is when the call's kernels start), maxima
// and sums of the rows on the diagonal tiles (2 B H n numbers), bf16 parts of K and V (6 B n H d each numbers of 16 bits, together).
struct F32Scratch {
    int* bad;
    int mark;
    float* ml;
    void* parts;
};
// The two kernels of attention on the tensor cores (psa_f32_attn_tensor.cu), for shapes that f32_tensor_attention_fits (psa_ws.h) and rows of 16 bytes.
cudaError_t f32_attention_split(const float* Q, const float* K, const float* V, const F32Scratch& fs, int B, int H, int n, int d, cudaStream_t stream);
cudaError_t f32_attention_tensor(const float* Q, float* out, const F32Scratch& fs, int B, int H, int n, int d, float scale, int masked, DeviceCounters* dc,
                                 cudaStream_t stream);
// Q, K, V, out: [B, n, H, d] fp32.  S: scratch [B*H, n, n] fp32, used by PSA_SYMMETRIC only.  fs: may be null.  dc_next (may be null): a second
// counter block, cleared by the last kernel.
cudaError_t f32_attention(const float* Q, const float* K, const float* V, float* out, float* S, const F32Scratch* fs, int B, int H,
                          int n, int d, float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next, cudaStream_t stream);

// Small layers in one launch (projections and the three phases of a (batch, head) per CTA, all in shared memory):
// f32_fused_fits says whether a shape qualifies.  X [B, n, D], W* [D, H*d] (Wk, Wv ignored for PSA_SYMMETRIC).
bool f32_fused_fits(int n, int D, int d, int scheme);
cudaError_t f32_fused_layer(const float* X, const float* Wq, const float* Wk, const float* Wv, float* out, int B, int H,
                            int n, int D, int d, float scale, int scheme, DeviceCounters* dc, DeviceCounters* dc_next,
                            cudaStream_t stream);   // (dc_next, if given, is cleared by the kernel for the next call)

// ---- bf16 tcgen05 path (psa_gemm.cu, psa_attn.cu) ----
// C[w][M, N] = A[M, K] * Bw[w][K, N] (+ residual[M, N], bf16, may be null), bf16 row-major, fp32 accumulation.
// Returns a psa_status.
int bf16_project(const void* A, const void* const Bw[3], void* const C[3], int nW, int M, int K, int N,
                 const void* residual, DeviceCounters* dc, cudaStream_t stream);
// Q, K, V, out: [B, n, H, d] bf16.  S: scratch for PSA_SYMMETRIC (sym_scratch_bytes:
// one 64 KB fp32 image per score block at or below the block diagonal, for the heads of one pass; with less, down to
// one head's worth, the call runs in more passes).
// `dc_next`, if not null, is a second counter block that the call's attention kernel clears (FULL, MASKED only).
// `cursor` is the work counter of the fused kernel (FULL, MASKED), zero when the call's kernels start.
// `s_clear`: bf16_symmetric_clear has been queued ahead of the call's kernels.
int bf16_attention(const void* Q, const void* K, const void* V, void* out, float* S, size_t s_bytes, bool s_clear, int B,
                   int H, int n, int d, float scale, int scheme, DeviceCounters* dc, unsigned int* cursor,
                   DeviceCounters* dc_next, cudaStream_t stream);
// Clears what the first pass of the symmetric kernel needs clear in its scratch, and `before` bytes ahead of the scratch.
cudaError_t bf16_symmetric_clear(float* S, size_t s_bytes, int B, int H, int n, size_t before, cudaStream_t stream);
// PSA_FULL and PSA_MASKED for 128 < d <= 256 (psa_attn_wide.cu).
int bf16_attention_wide(const void* Q, const void* K, const void* V, void* out, int B, int H, int n, int d, float scale,
                        int scheme, DeviceCounters* dc, unsigned int* cursor, DeviceCounters* dc_next, cudaStream_t stream);
// The persistent fused kernel behind bf16_attention for PSA_FULL and PSA_MASKED (psa_attn_persist.cu).
int bf16_attention_persist(const void* Q, const void* K, const void* V, void* out, int B, int H, int n, int d,
                           float scale, int scheme, DeviceCounters* dc, unsigned int* cursor, DeviceCounters* dc_next,
                           cudaStream_t stream);

// Once-per-device set-up of a kernel family.  Function attributes (the dynamic shared-memory limit) belong to the
// device that is current when they are set, and the SM count differs between devices, so both are kept per
// device ordinal.  device_setup() returns the current device's SM count (> 0), having run `configure` (which sets
// the family's attributes) the first time that device is seen; 0 on failure (error text set).  `device` (may be null): its ordinal.  Thread-safe.
constexpr int MAX_DEVICES = 64;
struct DeviceSetup {
    bool done[MAX_DEVICES];
    int sm_count[MAX_DEVICES];
};
int device_setup(DeviceSetup* st, cudaError_t (*configure)(), const char* what, int* device = nullptr);

// Self-test of the bounded-wait failure path (psa_selftest.cu): a one-CTA kernel whose barrier nobody completes.
cudaError_t launch_wait_expiry(DeviceCounters* dc, unsigned limit_us, cudaStream_t stream);

// Pipe-rate measurement (psa_pipes.cu): three kernels (ex2, fma, softmax mix), each storing per SM the cycles its
// slowest warp took for pipe_results_per_launch_per_sm() results.
cudaError_t launch_pipe_rates(unsigned long long* cycles, float* sink, int sms, cudaStream_t stream);
double pipe_results_per_launch_per_sm();

void set_cuda_error(cudaError_t e, const char* where);
void set_error_text(const char* text);

}  // namespace psa
