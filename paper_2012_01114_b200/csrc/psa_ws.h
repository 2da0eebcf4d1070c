// What lies where in the workspace of a call.  Host only, without CUDA, so that the layout can be checked on its own.
#pragma once
#include <stddef.h>
#include <string.h>

#include <algorithm>

#include "psa_sched.h"

namespace psa {

constexpr size_t COUNTER_BYTES = 256;          // counter blocks and cursors at the start of the workspace

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ---- which fp32 calls have scratch for the tensor cores
// Projection of [rows, D] by nW matrices [D, N], f32_project_pairs: bytes of bf16 parts of the operands (0: the call is not one of the
// largest ones, whatever the device), and number of marks.
inline size_t f32_project_parts_bytes(int rows, int D, int N, int nW) {
    const size_t tiles = (size_t)((rows + 255) / 256) * ((N + 255) / 256) * nW;
    if (D % 8 || N % 8 || tiles < 24 || (size_t)rows * D >= (size_t)1 << 33 || (size_t)D * N >= (size_t)1 << 33) return 0;
    return align_up((size_t)rows * D * 6, 256) + align_up((size_t)D * N * 6, 256) * nW;
}
inline size_t f32_project_marks(int rows, int N, int nW) { return (rows + 127) / 128 + (size_t)((N + 255) / 256) * nW; }
// Whether a projection may run there with `bytes` of room for its parts.  (A part of a call may ask for more than the call as a
// whole has: one with 2^33 numbers in X has no room for parts at all, a batch item of it would.)
inline bool f32_project_pairs_fit(int rows, int D, int N, int nW, size_t bytes) {
    const size_t need = f32_project_parts_bytes(rows, D, N, nW);
    return need != 0 && need <= bytes;
}

// Whether a call is better off on the tensor cores: three launches instead of one, and under the masked scheme a fourth for the diagonal
// tiles, which takes 20 to 30 us however few they are.  Measured at 4000 sizes at the edges; the CUDA cores' kernel moves in steps, with
// its rows per CTA (64, 32 or 16, by whether that makes two CTAs per SM) and slower where n is not a multiple of its 64 keys, and the diagonal
// tiles in rounds of one per SM (two up to d = 64).  Figures: heads, time on the tensor cores over time on CUDA cores.
// FULL: n = 129, d = 64 16 1.12; n = 160, d = 16 16 1.09, d = 64 16 0.89; n = 257, d = 16 8 1.08, 12 0.89; n = 256, d = 8 17 1.04, 20 0.88; n = 1024, d = 64 1 0.62.
// MASKED, up to 320 keys, where a head has three diagonal tiles and one or two blocks off them: d = 64 n = 257 32 1.33, 40 0.93, 64 0.58, n = 300 29 1.16, 32 0.84, n = 320
// 56 1.10, 79 0.82; d = 128 n = 257 29 1.04, 40 0.76, 53 1.12, 64 0.52; d = 32 n = 320 37 1.06, 63 0.78, n = 270 53 1.07; d = 8 n = 257 48 1.11, 64 0.80, 129 1.06,
// n = 320 53 1.31, 66 0.90, 123 1.22.  Beyond: d = 64 n = 385 22 1.07, 24 0.77, n = 420 20 1.06; d = 32 n = 385 22 1.12, 24 0.85; d = 8 n = 513 17 1.06, 20 0.82, n = 385 40 1.02;
// n = 640, d = 64 4 (100 blocks) 1.10, 12 0.86; n = 1024, d = 8 4 1.03, d = 64 4 0.80.
// Nor do calls come here whose error against 64 bits would be larger: with 16 rows per CTA the CUDA cores add up the keys in four chains, and for
// d > 80 on few keys that has less error than the tensor core's scores (FULL n = 192, d = 128 2.72e-7 and 2.80e-7, MASKED n = 385 2.07e-7 and 2.08e-7).
inline bool f32_tensor_attention_fits(int B, int H, int n, int d, int scheme) {
    constexpr int SMS = 148;
    const long long heads = (long long)B * H, T = row_tiles(n), tiles = heads * T, blocks = tiles * T;
    if (scheme == PSA_SYMMETRIC || d % 8 != 0 || heads * n * d >= (1LL << 31)) return false;
    const bool rows64 = heads * ((n + 63) / 64) >= 2 * SMS, rows32 = heads * ((n + 31) / 32) >= 2 * SMS;
    if (d > 80 && !rows32 && n <= (scheme == PSA_FULL ? 255 : 450)) return false;
    if (scheme == PSA_FULL)
        return n >= (d >= 64 ? 160 : 256) && blocks >= (d < 16 && n <= 256 ? 80 : 64) && (d >= 32 || heads * n * n >= 34LL * TILE * TILE);
    if (n <= 256 || blocks < (d >= 64 ? 256 : 320)) return false;
    if (n <= 320) {
        if (d > 64) return rows32 && (tiles <= SMS || rows64);
        return d >= 32 ? rows64 || (n % 64 != 0 && rows32 && tiles <= SMS) : rows64 && tiles <= 2 * SMS;
    }
    if (d > 64) return true;
    const long long off = heads * ((T - 1) * (T - 2) / 2 * TILE + (n - TILE * (T - 1)) * (T - 1));       // rows of 128 weights
    return (n > 576 || rows32) && (d >= 32 || off >= 100 * TILE);
}

// ---- the layout
// Scratch of the symmetric scheme in bf16: its heads in passes, see sym_heads_per_pass.
inline size_t sym_scratch_bytes(size_t heads, int n) {
    return (size_t)sym_heads_per_pass(heads, n, SYM_SCRATCH_CAP) * sym_pairs(row_tiles(n)) * S_BLOCK_BYTES;
}
struct WsShape {
    int batch, heads, n, d_model, d_k, scheme, dtype;
    bool with_proj, staging;       // projections ahead of the core; buffers of the host entry point
    bool one_launch;               // f32_fused_fits: a small fp32 layer, which needs no scratch but for an output projection
    bool lean;                     // without the scratch of the tensor cores: an fp32 call that has no memory for it runs on CUDA cores
};
struct WsLayout {
    size_t q, k, v, s, s_bytes, clear, clear_bytes, bad, marks_in, marks_pitch, marks_out, ml, parts, in_bytes, out_bytes, xs, wq, wk, wv, outs, total;
    bool attn_tensor;      // fp32: whether bad / ml / parts are there; in_bytes, out_bytes: room for the input and output projections' parts
};

inline WsLayout ws_layout(const WsShape& c) {
    const size_t es = c.dtype == PSA_BF16 ? 2 : 4;
    const size_t qkv = align_up((size_t)c.batch * c.n * c.heads * c.d_k * es, 256);
    const int rows = c.batch * c.n, hd = c.heads * c.d_k;
    WsLayout L;
    memset(&L, 0, sizeof(L));
    size_t off = COUNTER_BYTES;
    if (c.dtype == PSA_F32 && !c.lean) {      // marks right behind the counters: a captured call, the only one that clears marks, clears both in one go
        const size_t bh = (size_t)c.batch * c.heads;
        L.attn_tensor = !c.one_launch && f32_tensor_attention_fits(c.batch, c.heads, c.n, c.d_k, c.scheme);
        L.in_bytes = c.with_proj && !c.one_launch ? f32_project_parts_bytes(rows, c.d_model, hd, c.scheme == PSA_SYMMETRIC ? 1 : 3) : 0;
        L.out_bytes = c.with_proj ? f32_project_parts_bytes(rows, hd, c.d_model, 1) : 0;
        L.clear = off;
        if (L.attn_tensor) { L.bad = off; off += align_up(bh * sizeof(int), 256); }
        if (L.in_bytes) {      // (a part of a host call has marks of its own)
            L.marks_in = off; L.marks_pitch = f32_project_marks(rows, hd, 3);
            off += align_up((c.staging ? HOST_CHUNKS : 1) * L.marks_pitch * sizeof(int), 256);
        }
        if (L.out_bytes) { L.marks_out = off; off += align_up(f32_project_marks(rows, c.d_model, 1) * sizeof(int), 256); }
        L.clear_bytes = off - L.clear;
        if (L.attn_tensor) { L.ml = off; off += align_up(2 * bh * c.n * sizeof(float), 256); }
        L.parts = off;           // (used by one kernel after another)
        off += align_up(std::max(std::max(L.in_bytes, L.out_bytes), L.attn_tensor ? 12 * bh * c.n * c.d_k : (size_t)0), 256);
    }
    if (c.scheme == PSA_SYMMETRIC) {       // (bf16: right behind the counters, as above)
        L.s_bytes = c.dtype == PSA_BF16 ? sym_scratch_bytes((size_t)c.batch * c.heads, c.n) : align_up((size_t)c.batch * c.heads * c.n * c.n * sizeof(float), 256);
        L.s = off; off += L.s_bytes;
    }
    if (c.with_proj) {
        L.q = off; off += qkv;
        if (c.scheme == PSA_SYMMETRIC) { L.k = L.q; L.v = L.q; }
        else { L.k = off; off += qkv; L.v = off; off += qkv; }
    }
    if (c.staging) {
        const size_t xb = align_up((size_t)c.batch * c.n * c.d_model * es, 256);
        const size_t wb = align_up((size_t)c.d_model * c.heads * c.d_k * es, 256);
        L.xs = off; off += xb;
        L.wq = off; off += wb;
        if (c.scheme == PSA_SYMMETRIC) { L.wk = L.wq; L.wv = L.wq; }
        else { L.wk = off; off += wb; L.wv = off; off += wb; }
        L.outs = off; off += qkv;
    }
    L.total = off;
    return L;
}

// ---- which memory a call runs in: the caller's workspace, the library's own, or a new one of its own; and whether with the whole layout or
// the lean one.  A caller's workspace that holds the lean layout is used in any case: nothing is allocated behind the back of a
// caller who has registered one, and a graph keeps the memory that it was captured with.  `may_grow` is asked only where there is
// another way.
enum class WsFrom { USER, OWN, GROW };
struct WsPlan {
    WsFrom from;
    bool whole;
};
template <class MayGrow>
WsPlan ws_plan(size_t user, size_t own, size_t whole, size_t least, MayGrow may_grow) {
    if (user >= whole) return {WsFrom::USER, true};
    if (user >= least) return {WsFrom::USER, false};
    if (own >= whole) return {WsFrom::OWN, true};
    if (own >= least && !may_grow()) return {WsFrom::OWN, false};
    return {WsFrom::GROW, true};
}

}  // namespace psa
