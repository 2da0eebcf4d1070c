// Scratch of the symmetric scheme (paper Sec. 4), shared by its two kernels: sym_shared_kernel (psa_attn_sym.cu), which
// hands on weights, and sym_attn_kernel (psa_attn.cu), which hands on scores and takes any input.
//
// The scratch starts with a header of ints, cleared once per `heads` heads ahead of their first kernel:
//     [0] work counter of sym_shared_kernel   [1] number of heads it gave up
//     heads each: given up (0 / 1) | list of the heads given up | phase-1 blocks issued | phase-3 blocks issued |
//                 warps done with reading the head's blocks | work counters of sym_attn_kernel's launches
//     per head T ints, on cache lines of their own (148 CTAs look at them), each: blocks of tile I that sym_shared_kernel /
//                 sym_attn_kernel has handed on
// and holds the handed-on blocks behind it.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "psa_internal.h"
#include "psa_sched.h"
#include "sm100.cuh"

namespace psa {

constexpr int SYM_HEADER_WORDS = 16;
constexpr int SYM_PER_HEAD = 6;
constexpr int SYM_E_BYTES = 128 * 128 * 2;                      // a block of bf16 weights
constexpr int SYM_SUM_BYTES = 8 * 128 * 4;                      // its column sums, one row per 16 rows of the block
constexpr int SYM_SHARED_BLOCK_BYTES = SYM_E_BYTES + SYM_SUM_BYTES;

PSA_HD int sym_flag_pitch(int T) { return (T + 31) / 32 * 32; }
PSA_HD size_t sym_header_bytes(int heads, int T) {
    return (SYM_HEADER_WORDS + (size_t)SYM_PER_HEAD * heads + 32 + 2 * (size_t)heads * sym_flag_pitch(T)) * 4 / 1024 * 1024 + 1024;
}
struct SymHeader {
    int *work, *given_up, *bad, *list, *qk_blocks, *pv_blocks, *done, *general_work, *flags, *general_flags;
};
PSA_HD SymHeader sym_header(float* S, int heads, int T) {
    int* p = reinterpret_cast<int*>(S);
    SymHeader h;
    h.work = p; h.given_up = p + 1;
    p += SYM_HEADER_WORDS;
    h.bad = p; h.list = p + heads; h.qk_blocks = p + 2 * (size_t)heads; h.pv_blocks = p + 3 * (size_t)heads;
    h.done = p + 4 * (size_t)heads; h.general_work = p + 5 * (size_t)heads;
    p = reinterpret_cast<int*>(S) + (SYM_HEADER_WORDS + (size_t)SYM_PER_HEAD * heads + 31) / 32 * 32;
    h.flags = p; h.general_flags = p + (size_t)heads * sym_flag_pitch(T);
    return h;
}
// Blocks below the block diagonal of a head's weight matrix, numbered row by row.
PSA_HD size_t sym_lower_blocks(int T) { return (size_t)T * (T - 1) / 2; }
PSA_HD size_t sym_block_index(int I, int J) { return (size_t)I * (I - 1) / 2 + J; }

// Heads that one header serves: as many as leave the blocks of a pass (sym_heads_per_pass) their room in a scratch of `s_bytes`,
// which has 64 KB per row tile and head more than they take.
inline int sym_heads_per_header(size_t heads, int n, size_t s_bytes) {
    const size_t T = row_tiles(n), hp = sym_heads_per_pass(heads, n, s_bytes);
    const size_t fits = (hp * T * (S_BLOCK_BYTES / 2) - 2048) / ((SYM_PER_HEAD + 2 * (size_t)sym_flag_pitch((int)T)) * 4);
    return (int)(fits < heads ? fits : heads);
}

// One launch of sym_attn_kernel over `heads` heads from head bh0 on, or, given the list of heads that sym_shared_kernel gave
// up, over at most `heads` of them from entry `first` on.  `header_heads`: heads of the header; `launch`: number of this launch
// under that header.
int launch_sym_general(const void* X, void* out, float* S, int header_heads, int first, int heads, bool from_list, int launch, int bh0, int B, int H,
                       int n, int d, float scale, DeviceCounters* dc, cudaStream_t stream);
bool sym_shared_pays(int heads, int T, size_t s_bytes, int sms);
// sym_shared_kernel over `heads` heads from head bh0 on.
int launch_sym_shared(const void* X, void* out, float* S, size_t s_bytes, int heads, int bh0, int B, int H, int n, int d, float scale,
                      DeviceCounters* dc, cudaStream_t stream);

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

}  // namespace psa
