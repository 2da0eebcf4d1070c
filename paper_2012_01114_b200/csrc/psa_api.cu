// C interface of libpsa: argument checking, workspace management, the host twin of the tile
// scheduler (psa_skip_count) and dispatch to the fp32 and bf16 kernel families.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "psa_internal.h"
#include "psa_sched.h"
#include "psa_ws.h"

namespace psa {

namespace {

thread_local char g_err_text[256] = "";

// Marks of fp32 calls (heads and tiles that the tensor cores cannot take) are a number of the call's own, so that nothing has to be cleared ahead of
// its first kernel (us, with a clear ahead / without: layer of 4 x 512 x 768 85.1 / 81.2, core of 16 heads of n = 300, d = 128 24.6 / 21.3, of 32
// heads of n = 42 8.4 / 6.9).  What memory holds by chance or from an earlier call is another number; if it is the same after all, a head or
// tile is worked on by the path for marked ones, which takes any.
constexpr int MARK_BASE = 0x5a000000;

struct Context {
    std::mutex mu;
    void* user_ws = nullptr;
    size_t user_bytes = 0;
    void* own_ws = nullptr;
    size_t own_bytes = 0;
    DeviceCounters* last_dc = nullptr;  // counters of the most recent call
    // The workspace starts with three counter blocks.  All paths but the symmetric one in bf16 use the first two in turn: the
    // last attention kernel of a call clears the block of the next call, so that no clearing copy has to run ahead of the
    // call's first kernel.  `clean_ws` is the workspace whose block `next_block` is known to be clear.  A call that is being
    // captured into a graph has the third to itself and clears it first: the graph may run any number of times, between
    // any other calls.
    char* clean_ws = nullptr;
    int next_block = 0;
    int mark = MARK_BASE;               // see next_mark
    // Streams and events of the entry points on host buffers, created by the first such call and kept.
    struct HostPipe* pipe = nullptr;
    std::vector<cudaEvent_t> prof_events;  // 3 per profiled call
    int prof_calls = 0, prof_max = 0;
    psa_counts last_useful = {0, 0, 0, 0, 0, 0};
};
// One context per device ordinal: workspace, counters and profiling state belong to the device that was current
// when they were created.  Every entry point works on the context of the calling thread's current device.
Context g_ctxs[MAX_DEVICES];
std::mutex g_setup_mu;

Context* current_ctx() {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { set_cuda_error(e, "cudaGetDevice"); return nullptr; }
    if (dev < 0 || dev >= MAX_DEVICES) { set_error_text("device ordinal beyond the library's table"); return nullptr; }
    return &g_ctxs[dev];
}

struct HostPipe {
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t start = nullptr, loaded[HOST_CHUNKS] = {}, computed[HOST_CHUNKS] = {}, stored = nullptr;
};

constexpr size_t COUNTER_BLOCK_BYTES = 64;
constexpr int TURN_BLOCKS = 2, CAPTURE_BLOCK = 2;      // blocks used in turn; block of captured calls
constexpr size_t CURSOR_OFFSET = 3 * COUNTER_BLOCK_BYTES;   // work counters of a call in several parts
static_assert(sizeof(DeviceCounters) <= COUNTER_BLOCK_BYTES, "counter block too small");
static_assert(CURSOR_OFFSET + HOST_CHUNKS * sizeof(unsigned int) <= COUNTER_BYTES, "no room for the cursors");

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_shape(int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, bool with_proj) {
    if (scheme != PSA_FULL && scheme != PSA_SYMMETRIC && scheme != PSA_MASKED) return PSA_ERR_SCHEME_ARGS;
    if (dtype != PSA_F32 && dtype != PSA_BF16) return PSA_ERR_UNSUPPORTED;
    if (batch <= 0 || heads <= 0 || n <= 0 || d_k <= 0 || (with_proj && d_model <= 0)) return PSA_ERR_SHAPE;
    if ((double)batch * heads * n * (double)d_k > 4.0e12 || (double)batch * n * (double)(with_proj ? d_model : 1) > 4.0e12)
        return PSA_ERR_SHAPE;
    if ((long long)batch * n > 0x7fffffffLL || (long long)heads * d_k > 0x7fffffffLL) return PSA_ERR_SHAPE;
    if (dtype == PSA_BF16) {
        // heads of up to 256 columns for the full and masked schemes; the symmetric scheme's kernels stop at 128
        if (d_k < 8 || d_k > (scheme == PSA_SYMMETRIC ? 128 : 256) || d_k % 8 != 0) return PSA_ERR_UNSUPPORTED;
        if (with_proj && (d_model % 64 != 0)) return PSA_ERR_UNSUPPORTED;
    } else {
        if (n > 1024 || d_k > 128) return PSA_ERR_UNSUPPORTED;
    }
    return PSA_OK;
}

WsShape call_shape(int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, bool with_proj, bool staging) {
    return WsShape{batch, heads, n, d_model, d_k, scheme, dtype, with_proj, staging, with_proj && dtype == PSA_F32 && f32_fused_fits(n, d_model, d_k, scheme), false};
}

int next_mark(Context& cx) { return cx.mark = cx.mark == 0x7fffffff ? MARK_BASE : cx.mark + 1; }

F32Scratch f32_scratch(char* ws, const WsLayout& L, size_t first_head, int mark) {
    return F32Scratch{reinterpret_cast<int*>(ws + L.bad) + first_head, mark, reinterpret_cast<float*>(ws + L.ml), ws + L.parts};
}

// Whether copies from or to this host memory run beside the calling thread (memory that CUDA knows of).
bool pinned(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) == cudaSuccess) return a.type != cudaMemoryTypeUnregistered;
    cudaGetLastError();
    return false;
}

HostPipe* acquire_pipe(Context& cx) {
    if (cx.pipe) return cx.pipe;
    HostPipe* p = new (std::nothrow) HostPipe;
    if (!p) { set_error_text("out of host memory"); return nullptr; }
    cudaError_t e = cudaStreamCreateWithFlags(&p->in, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->out, cudaStreamNonBlocking);
    auto event = [&](cudaEvent_t* ev) { if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming); };
    event(&p->start); event(&p->stored);
    for (int c = 0; c < HOST_CHUNKS; ++c) { event(&p->loaded[c]); event(&p->computed[c]); }
    if (e == cudaSuccess) return cx.pipe = p;
    set_cuda_error(e, "streams of the host entry points");
    if (p->in) cudaStreamDestroy(p->in);
    if (p->out) cudaStreamDestroy(p->out);
    for (cudaEvent_t ev : {p->start, p->stored}) if (ev) cudaEventDestroy(ev);
    for (int c = 0; c < HOST_CHUNKS; ++c) {
        if (p->loaded[c]) cudaEventDestroy(p->loaded[c]);
        if (p->computed[c]) cudaEventDestroy(p->computed[c]);
    }
    delete p;
    return nullptr;
}

// Replaces the library's own workspace.  nullptr (error text set) if there is no memory.
char* grow_ws(Context& cx, size_t bytes) {
    if (cx.own_ws) {
        cudaDeviceSynchronize();
        cudaFree(cx.own_ws);
        cx.own_ws = nullptr;
        cx.own_bytes = 0;
        cx.last_dc = nullptr;       // (may have been in it)
    }
    void* p = nullptr;
    const cudaError_t e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) {
        set_cuda_error(e, "cudaMalloc(workspace)");
        cudaGetLastError();         // (the next launch must not find it)
        return nullptr;
    }
    cx.own_ws = p;
    cx.clean_ws = nullptr;          // fresh memory: no counter block is known to be clear
    cx.own_bytes = bytes;
    return static_cast<char*>(p);
}

// Returns the base of a workspace of at least `bytes`, or nullptr (error text set).
char* acquire_ws(Context& cx, size_t bytes) {
    if (cx.user_ws && cx.user_bytes >= bytes) return static_cast<char*>(cx.user_ws);
    if (cx.own_ws && cx.own_bytes >= bytes) return static_cast<char*>(cx.own_ws);
    return grow_ws(cx, bytes);
}

// The workspace of a call and what lies where in it, `extra` bytes behind the layout (from L->total on) included; nullptr (error text set) if
// there is none.  fp32 calls do with the lean layout where the whole one finds no memory.
char* acquire_call_ws(Context& cx, WsShape c, size_t extra, cudaStream_t stream, WsLayout* L) {
    *L = ws_layout(c);
    const size_t whole = L->total + extra, user = cx.user_ws ? cx.user_bytes : 0, own = cx.own_ws ? cx.own_bytes : 0;
    if (c.dtype != PSA_F32 || user >= whole || (!user && own >= whole)) return acquire_ws(cx, whole);
    c.lean = true;
    const WsLayout lean = ws_layout(c);
    const size_t least = lean.total + extra;
    const WsPlan plan = ws_plan(user, own, whole, least, [&] {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        size_t avail = 0, total = 0;
        return cudaStreamIsCapturing(stream, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone &&
               cudaMemGetInfo(&avail, &total) == cudaSuccess && avail + own >= whole;
    });
    char* ws = static_cast<char*>(plan.from == WsFrom::USER ? cx.user_ws : cx.own_ws);
    bool use_lean = !plan.whole;
    if (plan.from == WsFrom::GROW) {
        ws = grow_ws(cx, whole);
        if (!ws && least < whole) {
            ws = grow_ws(cx, least);
            if (ws) g_err_text[0] = 0;
            use_lean = true;
        }
    }
    if (use_lean) *L = lean;
    return ws;
}

void useful_counts(int batch, int heads, int n, int d_model, int d_k, int scheme, bool with_proj, psa_counts* c) {
    const uint64_t bh = (uint64_t)batch * heads, N = n, d = d_k;
    const uint64_t tri = N * (N + 1) / 2;
    c->useful_qk_macs = bh * d * (scheme == PSA_FULL ? N * N : tri);
    c->useful_pv_macs = bh * d * (scheme == PSA_MASKED ? tri : N * N);
    const uint64_t nproj = scheme == PSA_SYMMETRIC ? 1 : 3;
    c->proj_macs = with_proj ? nproj * (uint64_t)batch * N * (uint64_t)d_model * (uint64_t)heads * d : 0;
}

// The kernels of one layer (or, without projections, of one attention core) over `batch` sequences.  q, k, v: the workspace's
// projections (with_proj), written here; `cursor`: work counter of the fused bf16 kernel, zero when it starts; `dc_next`: see
// Context (may be null).  `between`, if given, is recorded between projections and attention.
int enqueue_layer(const void* X, const void* Wq, const void* Wk, const void* Wv, const void* Q, const void* K, const void* V,
                  int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, void* out, cudaStream_t stream,
                  bool with_proj, void* const qkv[3], float* S, size_t s_bytes, bool s_clear, const F32Scratch* fs, const F32ProjectScratch* ps,
                  DeviceCounters* dc, unsigned int* cursor,
                  DeviceCounters* dc_next, cudaEvent_t between) {
    const float scale = 1.0f / sqrtf((float)d_k);
    const int nW = scheme == PSA_SYMMETRIC ? 1 : 3;
    cudaError_t e = cudaSuccess;
    if (with_proj && dtype == PSA_F32 && f32_fused_fits(n, d_model, d_k, scheme)) {
        // a small fp32 layer runs as one launch; q, k, v never leave shared memory
        if (between) cudaEventRecord(between, stream);
        e = f32_fused_layer(static_cast<const float*>(X), static_cast<const float*>(Wq), static_cast<const float*>(Wk),
                            static_cast<const float*>(Wv), static_cast<float*>(out), batch, heads, n, d_model, d_k, scale,
                            scheme, dc, dc_next, stream);
        if (e != cudaSuccess) { set_cuda_error(e, "f32_fused_layer"); return PSA_ERR_CUDA; }
        return PSA_OK;
    }
    if (with_proj) {
        const void* Ws[3] = {Wq, nW == 3 ? Wk : Wq, nW == 3 ? Wv : Wq};
        if (dtype == PSA_F32) {
            float* const outs[3] = {static_cast<float*>(qkv[0]), static_cast<float*>(qkv[1]), static_cast<float*>(qkv[2])};
            e = f32_project(static_cast<const float*>(X), reinterpret_cast<const float* const*>(Ws), outs, nW, batch * n, d_model,
                            heads * d_k, nullptr, ps, dc, stream);
            if (e != cudaSuccess) { set_cuda_error(e, "f32_project"); return PSA_ERR_CUDA; }
        } else {
            int rc = bf16_project(X, Ws, qkv, nW, batch * n, d_model, heads * d_k, nullptr, dc, stream);
            if (rc != PSA_OK) return rc;
        }
        Q = qkv[0]; K = qkv[1]; V = qkv[2];
    }
    if (between) cudaEventRecord(between, stream);
    if (dtype == PSA_F32) {
        e = f32_attention(static_cast<const float*>(Q), static_cast<const float*>(K), static_cast<const float*>(V),
                          static_cast<float*>(out), S, fs, batch, heads, n, d_k, scale, scheme, dc, dc_next, stream);
        if (e != cudaSuccess) { set_cuda_error(e, "f32_attention"); return PSA_ERR_CUDA; }
        return PSA_OK;
    }
    return bf16_attention(Q, K, V, out, S, s_bytes, s_clear, batch, heads, n, d_k, scale, scheme, dc, cursor, dc_next, stream);
}

int run_layer(Context& cx, const void* X, const void* Wq, const void* Wk, const void* Wv, const void* Q, const void* K,
              const void* V, int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, void* out,
              cudaStream_t stream, bool with_proj, char* ws, const WsLayout& L) {
    // the paths whose last attention kernel clears the other counter block
    const bool turns = dtype == PSA_F32 || scheme != PSA_SYMMETRIC;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &capture);
    if (e != cudaSuccess) { set_cuda_error(e, "cudaStreamIsCapturing"); return PSA_ERR_CUDA; }
    const bool captured = capture != cudaStreamCaptureStatusNone;
    float* S = scheme == PSA_SYMMETRIC ? reinterpret_cast<float*>(ws + L.s) : nullptr;
    const bool s_clear = !captured && S && dtype == PSA_BF16;      // counters and flags of the symmetric kernel cleared in one go
    int block = 0;
    if (captured) {
        block = CAPTURE_BLOCK;
        // (its mark stays the same in every replay, so that marks are cleared too; the cursors between are those of host calls, which clear them)
        const size_t first = CAPTURE_BLOCK * COUNTER_BLOCK_BYTES;
        e = cudaMemsetAsync(ws + first, 0, (L.clear_bytes ? L.clear + L.clear_bytes : first + COUNTER_BLOCK_BYTES) - first, stream);
    } else if (s_clear) {
        e = bf16_symmetric_clear(S, L.s_bytes, batch, heads, n, L.s, stream);
    } else if (turns && cx.clean_ws == ws) {
        block = cx.next_block;
    } else {
        e = cudaMemsetAsync(ws, 0, TURN_BLOCKS * COUNTER_BLOCK_BYTES, stream);
    }
    if (e != cudaSuccess) { set_cuda_error(e, "cudaMemsetAsync(counters)"); return PSA_ERR_CUDA; }
    if (!captured) cx.clean_ws = nullptr;          // until this call's kernels are known to be queued
    DeviceCounters* dc = reinterpret_cast<DeviceCounters*>(ws + block * COUNTER_BLOCK_BYTES);
    DeviceCounters* dc_next = turns && !captured ? reinterpret_cast<DeviceCounters*>(ws + (block ^ 1) * COUNTER_BLOCK_BYTES) : nullptr;
    cx.last_dc = dc;
    memset(&cx.last_useful, 0, sizeof(psa_counts));
    useful_counts(batch, heads, n, d_model, d_k, scheme, with_proj, &cx.last_useful);
    cudaEvent_t* pev = nullptr;
    if (cx.prof_calls < cx.prof_max) pev = &cx.prof_events[3 * cx.prof_calls++];
    struct EventTail {  // records the closing event on every exit path
        cudaEvent_t* ev; cudaStream_t st;
        ~EventTail() { if (ev) cudaEventRecord(ev[2], st); }
    } tail{pev, stream};
    if (pev) cudaEventRecord(pev[0], stream);
    void* const qkv[3] = {ws + L.q, ws + L.k, ws + L.v};
    const int mark = next_mark(cx);
    const F32Scratch fs = f32_scratch(ws, L, 0, mark);
    const F32ProjectScratch ps = {ws + L.parts, L.in_bytes, reinterpret_cast<int*>(ws + L.marks_in), mark};
    const int rc = enqueue_layer(X, Wq, Wk, Wv, Q, K, V, batch, heads, n, d_model, d_k, scheme, dtype, out, stream, with_proj,
                                 qkv, S, L.s_bytes, s_clear, L.attn_tensor ? &fs : nullptr, L.in_bytes ? &ps : nullptr, dc, &dc->next_item, dc_next, pev ? pev[1] : nullptr);
    if (rc == PSA_OK && turns && !captured) {        // the other block will be clear once this call has run
        cx.clean_ws = ws;
        cx.next_block = block ^ 1;
    }
    return rc;
}

int layer_entry(const void* X, const void* Wq, const void* Wk, const void* Wv, int batch, int heads, int n,
                int d_model, int d_k, int scheme, int dtype, void* out, void* stream) {
    g_err_text[0] = 0;
    int rc = check_shape(batch, heads, n, d_model, d_k, scheme, dtype, true);
    if (rc != PSA_OK) return rc;
    if (!X || !Wq || !out) return PSA_ERR_NULL;
    if (scheme == PSA_SYMMETRIC) {
        if ((Wk && Wk != Wq) || (Wv && Wv != Wq)) return PSA_ERR_SCHEME_ARGS;
    } else if (!Wk || !Wv) {
        return PSA_ERR_NULL;
    }
    if (!aligned16(X) || !aligned16(Wq) || !aligned16(Wk) || !aligned16(Wv) || !aligned16(out)) return PSA_ERR_ALIGN;
    if (dtype == PSA_BF16 && (heads * d_k) % 64 != 0) return PSA_ERR_UNSUPPORTED;
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    WsLayout L;
    char* ws = acquire_call_ws(cx, call_shape(batch, heads, n, d_model, d_k, scheme, dtype, true, false), 0, static_cast<cudaStream_t>(stream), &L);
    if (!ws) return PSA_ERR_WORKSPACE;
    return run_layer(cx, X, Wq, Wk, Wv, nullptr, nullptr, nullptr, batch, heads, n, d_model, d_k, scheme, dtype, out,
                     static_cast<cudaStream_t>(stream), true, ws, L);
}

}  // namespace

int device_setup(DeviceSetup* st, cudaError_t (*configure)(), const char* what, int* device) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) { set_cuda_error(e, what); return 0; }
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (!st->done[dev]) {
        int sms = 0;
        e = configure();
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess || sms <= 0) { set_cuda_error(e, what); return 0; }
        st->sm_count[dev] = sms;
        st->done[dev] = true;
    }
    if (device) *device = dev;
    return st->sm_count[dev];
}

void set_cuda_error(cudaError_t e, const char* where) {
    snprintf(g_err_text, sizeof(g_err_text), "%s: %s", where, cudaGetErrorString(e));
}
void set_error_text(const char* text) { snprintf(g_err_text, sizeof(g_err_text), "%s", text); }

}  // namespace psa

using namespace psa;

extern "C" {

int psa_attention(const void* X, const void* Wq, const void* Wk, const void* Wv, int batch, int heads, int n,
                  int d_model, int d_k, int scheme, void* out, void* stream) {
    return layer_entry(X, Wq, Wk, Wv, batch, heads, n, d_model, d_k, scheme, PSA_BF16, out, stream);
}

int psa_attention_f32(const void* X, const void* Wq, const void* Wk, const void* Wv, int batch, int heads, int n,
                      int d_model, int d_k, int scheme, void* out, void* stream) {
    return layer_entry(X, Wq, Wk, Wv, batch, heads, n, d_model, d_k, scheme, PSA_F32, out, stream);
}

int psa_attention_core(const void* Q, const void* K, const void* V, int batch, int heads, int n, int d_k,
                       int scheme, int dtype, void* out, void* stream) {
    g_err_text[0] = 0;
    int rc = check_shape(batch, heads, n, 0, d_k, scheme, dtype, false);
    if (rc != PSA_OK) return rc;
    if (!Q || !out) return PSA_ERR_NULL;
    if (scheme == PSA_SYMMETRIC) {
        if ((K && K != Q) || (V && V != Q)) return PSA_ERR_SCHEME_ARGS;
        K = Q; V = Q;
    } else if (!K || !V) {
        return PSA_ERR_NULL;
    }
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(out)) return PSA_ERR_ALIGN;
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    WsLayout L;
    char* ws = acquire_call_ws(cx, call_shape(batch, heads, n, 0, d_k, scheme, dtype, false, false), 0, static_cast<cudaStream_t>(stream), &L);
    if (!ws) return PSA_ERR_WORKSPACE;
    // In place (fp32): the CUDA-core kernels read a row of Q before they write it, as the tensor-core one of the full scheme does; the masked
    // one keeps partial outputs in `out` while Q is still to be read.
    const uintptr_t q0 = reinterpret_cast<uintptr_t>(Q), o0 = reinterpret_cast<uintptr_t>(out), bytes = (uintptr_t)batch * n * heads * d_k * 4;
    if (dtype == PSA_F32 && scheme == PSA_MASKED && q0 < o0 + bytes && o0 < q0 + bytes) L.attn_tensor = false;
    return run_layer(cx, nullptr, nullptr, nullptr, nullptr, Q, K, V, batch, heads, n, 0, d_k, scheme, dtype, out,
                     static_cast<cudaStream_t>(stream), false, ws, L);
}

int psa_attention_host(const void* X_host, const void* Wq_host, const void* Wk_host, const void* Wv_host,
                       int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, void* out_host,
                       void* stream_v) {
    g_err_text[0] = 0;
    int rc = check_shape(batch, heads, n, d_model, d_k, scheme, dtype, true);
    if (rc != PSA_OK) return rc;
    if (!X_host || !Wq_host || !out_host) return PSA_ERR_NULL;
    if (scheme == PSA_SYMMETRIC) {
        if ((Wk_host && Wk_host != Wq_host) || (Wv_host && Wv_host != Wq_host)) return PSA_ERR_SCHEME_ARGS;
    } else if (!Wk_host || !Wv_host) {
        return PSA_ERR_NULL;
    }
    if (dtype == PSA_BF16 && (heads * d_k) % 64 != 0) return PSA_ERR_UNSUPPORTED;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    WsLayout L;
    char* ws = acquire_call_ws(cx, call_shape(batch, heads, n, d_model, d_k, scheme, dtype, true, true), 0, stream, &L);
    if (!ws) return PSA_ERR_WORKSPACE;
    const size_t es = dtype == PSA_BF16 ? 2 : 4;
    const size_t xb = (size_t)n * d_model * es, wb = (size_t)d_model * heads * d_k * es, ob = (size_t)n * heads * d_k * es;   // per sequence; per matrix
    int parts = host_parts(batch, xb, ob, X_host, out_host);
    HostPipe* pipe = nullptr;
    if (parts > 1 && cx.prof_calls >= cx.prof_max) {         // (a call that is being timed runs in one part, on one stream)
        pipe = acquire_pipe(cx);
        if (!pipe) return PSA_ERR_CUDA;
    }
    const bool sym = scheme == PSA_SYMMETRIC;
    if (!pipe) {
        cudaError_t e = cudaMemcpyAsync(ws + L.xs, X_host, batch * xb, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.wq, Wq_host, wb, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess && !sym) {
            e = cudaMemcpyAsync(ws + L.wk, Wk_host, wb, cudaMemcpyHostToDevice, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.wv, Wv_host, wb, cudaMemcpyHostToDevice, stream);
        }
        if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync(H2D)"); return PSA_ERR_CUDA; }
        rc = run_layer(cx, ws + L.xs, ws + L.wq, ws + L.wk, ws + L.wv, nullptr, nullptr, nullptr, batch, heads, n, d_model,
                       d_k, scheme, dtype, ws + L.outs, stream, true, ws, L);
        if (rc != PSA_OK) return rc;
        e = cudaMemcpyAsync(out_host, ws + L.outs, batch * ob, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync(D2H)/sync"); return PSA_ERR_CUDA; }
        return PSA_OK;
    }
    // In parts: copies in on one stream, kernels on the caller's, copies out on another.  The counters of all parts go to one
    // block; the work counter of each has a place of its own behind the blocks.  All copies in are queued before the first copy
    // out: one from pageable memory (a matrix) holds the calling thread until it is done.
    const char* what = "ordering the streams of a host call";
    cudaError_t e = cudaEventRecord(pipe->start, stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe->in, pipe->start, 0);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe->out, pipe->start, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, COUNTER_BYTES, stream);
    cx.clean_ws = nullptr;
    DeviceCounters* dc = reinterpret_cast<DeviceCounters*>(ws);
    cx.last_dc = dc;
    memset(&cx.last_useful, 0, sizeof(psa_counts));
    useful_counts(batch, heads, n, d_model, d_k, scheme, true, &cx.last_useful);
    if (e == cudaSuccess) {
        what = "cudaMemcpyAsync(H2D)";
        e = cudaMemcpyAsync(ws + L.wq, Wq_host, wb, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess && !sym) e = cudaMemcpyAsync(ws + L.wk, Wk_host, wb, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess && !sym) e = cudaMemcpyAsync(ws + L.wv, Wv_host, wb, cudaMemcpyHostToDevice, pipe->in);
    }
    // One part for bf16 in pageable buffers: copies from and to these hold the calling thread, so that little overlaps, and every
    // further copy costs (16 x 512 x 768, 12 heads: 1597 us in one part, 1812 in eight; in fp32, whose kernels take longer, 4140
    // and 3310).  Asked here, under the copies of the matrices: the answer takes a few microseconds per buffer.
    if (dtype == PSA_BF16 && !(pinned(X_host) && pinned(out_host))) parts = 1;
    const int mark = next_mark(cx);
    auto first = [&](int c) { return (int)((long long)batch * c / parts); };      // first sequence of part c
    for (int c = 0; c < parts && e == cudaSuccess; ++c) {
        const size_t b0 = first(c), nb = first(c + 1) - b0;
        e = cudaMemcpyAsync(ws + L.xs + b0 * xb, static_cast<const char*>(X_host) + b0 * xb, nb * xb, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess) e = cudaEventRecord(pipe->loaded[c], pipe->in);
    }
    for (int c = 0; c < parts && e == cudaSuccess && rc == PSA_OK; ++c) {
        const size_t b0 = first(c), nb = first(c + 1) - b0;
        what = "ordering the streams of a host call";
        e = cudaStreamWaitEvent(stream, pipe->loaded[c], 0);
        if (e != cudaSuccess) break;
        void* const qkv[3] = {ws + L.q + b0 * ob, ws + L.k + b0 * ob, ws + L.v + b0 * ob};
        const F32ProjectScratch ps = {ws + L.parts, L.in_bytes, reinterpret_cast<int*>(ws + L.marks_in) + c * L.marks_pitch, mark};
        const F32Scratch fs = f32_scratch(ws, L, b0 * heads, mark);       // (a part has marks of its own; the rest is used by one after another)
        rc = enqueue_layer(ws + L.xs + b0 * xb, ws + L.wq, ws + L.wk, ws + L.wv, nullptr, nullptr, nullptr, (int)nb, heads, n, d_model,
                           d_k, scheme, dtype, ws + L.outs + b0 * ob, stream, true, qkv,
                           sym ? reinterpret_cast<float*>(ws + L.s) : nullptr, L.s_bytes, false, L.attn_tensor ? &fs : nullptr, L.in_bytes ? &ps : nullptr, dc,
                           reinterpret_cast<unsigned int*>(ws + CURSOR_OFFSET) + c, nullptr, nullptr);
        if (rc != PSA_OK) break;
        e = cudaEventRecord(pipe->computed[c], stream);
    }
    for (int c = 0; c < parts && e == cudaSuccess && rc == PSA_OK; ++c) {
        const size_t b0 = first(c), nb = first(c + 1) - b0;
        what = "cudaMemcpyAsync(D2H)";
        e = cudaStreamWaitEvent(pipe->out, pipe->computed[c], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(static_cast<char*>(out_host) + b0 * ob, ws + L.outs + b0 * ob, nb * ob, cudaMemcpyDeviceToHost, pipe->out);
    }
    if (e == cudaSuccess && rc == PSA_OK) e = cudaEventRecord(pipe->stored, pipe->out);
    if (e == cudaSuccess && rc == PSA_OK) e = cudaStreamWaitEvent(stream, pipe->stored, 0);
    if (e == cudaSuccess && rc == PSA_OK) {
        e = cudaStreamSynchronize(stream);
    } else {            // nothing of this call may touch the caller's buffers after it has returned
        cudaStreamSynchronize(pipe->in);
        cudaStreamSynchronize(stream);
        cudaStreamSynchronize(pipe->out);
    }
    if (rc != PSA_OK) return rc;
    if (e != cudaSuccess) { set_cuda_error(e, what); return PSA_ERR_CUDA; }
    return PSA_OK;
}

int psa_attention_core_host(const void* Q_host, const void* K_host, const void* V_host, int batch, int heads, int n,
                            int d_k, int scheme, int dtype, void* out_host, void* stream_v) {
    g_err_text[0] = 0;
    int rc = check_shape(batch, heads, n, 0, d_k, scheme, dtype, false);
    if (rc != PSA_OK) return rc;
    if (!Q_host || !out_host) return PSA_ERR_NULL;
    const bool sym = scheme == PSA_SYMMETRIC;
    if (sym) {
        if ((K_host && K_host != Q_host) || (V_host && V_host != Q_host)) return PSA_ERR_SCHEME_ARGS;
    } else if (!K_host || !V_host) {
        return PSA_ERR_NULL;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    const size_t tb = (size_t)batch * n * heads * d_k * (dtype == PSA_BF16 ? 2 : 4), tba = align_up(tb, 256);
    WsLayout L;
    char* ws = acquire_call_ws(cx, call_shape(batch, heads, n, 0, d_k, scheme, dtype, false, false), (sym ? 2 : 4) * tba, stream, &L);
    if (!ws) return PSA_ERR_WORKSPACE;
    const size_t q_off = L.total, k_off = q_off + tba, v_off = k_off + tba;
    const size_t o_off = sym ? k_off : v_off + tba;          // the symmetric scheme stages one input tensor
    cudaError_t e = cudaMemcpyAsync(ws + q_off, Q_host, tb, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess && !sym) {
        e = cudaMemcpyAsync(ws + k_off, K_host, tb, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ws + v_off, V_host, tb, cudaMemcpyHostToDevice, stream);
    }
    if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync(H2D)"); return PSA_ERR_CUDA; }
    const void* q = ws + q_off;
    rc = run_layer(cx, nullptr, nullptr, nullptr, nullptr, q, sym ? q : ws + k_off, sym ? q : ws + v_off, batch, heads, n,
                   0, d_k, scheme, dtype, ws + o_off, stream, false, ws, L);
    if (rc != PSA_OK) return rc;
    e = cudaMemcpyAsync(out_host, ws + o_off, tb, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) { set_cuda_error(e, "cudaMemcpyAsync(D2H)/sync"); return PSA_ERR_CUDA; }
    return PSA_OK;
}

int psa_attention_block(const void* X, const void* Wq, const void* Wk, const void* Wv, const void* Wo, int batch,
                        int heads, int n, int d_model, int d_k, int scheme, int dtype, void* out, void* stream_v) {
    return psa_attention_block_residual(X, Wq, Wk, Wv, Wo, nullptr, batch, heads, n, d_model, d_k, scheme, dtype, out,
                                        stream_v);
}

int psa_attention_block_residual(const void* X, const void* Wq, const void* Wk, const void* Wv, const void* Wo,
                                 const void* R, int batch, int heads, int n, int d_model, int d_k, int scheme,
                                 int dtype, void* out, void* stream_v) {
    g_err_text[0] = 0;
    int rc = check_shape(batch, heads, n, d_model, d_k, scheme, dtype, true);
    if (rc != PSA_OK) return rc;
    if (!X || !Wq || !Wo || !out) return PSA_ERR_NULL;
    if (scheme == PSA_SYMMETRIC) {
        if ((Wk && Wk != Wq) || (Wv && Wv != Wq)) return PSA_ERR_SCHEME_ARGS;
    } else if (!Wk || !Wv) {
        return PSA_ERR_NULL;
    }
    if (!aligned16(X) || !aligned16(Wq) || !aligned16(Wk) || !aligned16(Wv) || !aligned16(Wo) || !aligned16(out) ||
        !aligned16(R))
        return PSA_ERR_ALIGN;
    if (R == out) return PSA_ERR_SCHEME_ARGS;      // the residual is read while the output is written
    if (dtype == PSA_BF16 && (heads * d_k) % 64 != 0) return PSA_ERR_UNSUPPORTED;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    WsLayout L;
    char* ws = acquire_call_ws(cx, call_shape(batch, heads, n, d_model, d_k, scheme, dtype, true, false), align_up((size_t)batch * n * heads * d_k * (dtype == PSA_BF16 ? 2 : 4), 256),
                               stream, &L);
    if (!ws) return PSA_ERR_WORKSPACE;
    void* y = ws + L.total;
    rc = run_layer(cx, X, Wq, Wk, Wv, nullptr, nullptr, nullptr, batch, heads, n, d_model, d_k, scheme, dtype, y, stream,
                   true, ws, L);
    if (rc != PSA_OK) return rc;
    // z = y * Wo with the projection kernel; its MACs are added to the call's counter block
    const void* Ws[3] = {Wo, Wo, Wo};
    void* outs[3] = {out, out, out};
    if (dtype == PSA_F32) {
        const F32ProjectScratch ps = {ws + L.parts, L.out_bytes, reinterpret_cast<int*>(ws + L.marks_out), cx.mark};
        const cudaError_t e = f32_project(static_cast<const float*>(y), reinterpret_cast<const float* const*>(Ws),
                                          reinterpret_cast<float* const*>(outs), 1, batch * n, heads * d_k, d_model,
                                          static_cast<const float*>(R), L.out_bytes ? &ps : nullptr, cx.last_dc, stream);
        if (e != cudaSuccess) { set_cuda_error(e, "f32_project(Wo)"); return PSA_ERR_CUDA; }
        return PSA_OK;
    }
    return bf16_project(y, Ws, outs, 1, batch * n, heads * d_k, d_model, R, cx.last_dc, stream);
}

size_t psa_block_workspace_bytes(int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype) {
    if (d_model <= 0 || check_shape(batch, heads, n, d_model, d_k, scheme, dtype, true) != PSA_OK) return 0;
    return ws_layout(call_shape(batch, heads, n, d_model, d_k, scheme, dtype, true, false)).total + align_up((size_t)batch * n * heads * d_k * (dtype == PSA_BF16 ? 2 : 4), 256);
}

int psa_skip_count(int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype, psa_counts* c) {
    if (!c) return PSA_ERR_NULL;
    const bool with_proj = d_model > 0;
    int rc = check_shape(batch, heads, n, d_model, d_k, scheme, dtype, with_proj);
    if (rc != PSA_OK) return rc;
    memset(c, 0, sizeof(*c));
    useful_counts(batch, heads, n, d_model, d_k, scheme, with_proj, c);
    const uint64_t bh = (uint64_t)batch * heads;
    if (dtype == PSA_F32) {  // element-exact skipping
        c->qk_macs = c->useful_qk_macs;
        c->pv_macs = c->useful_pv_macs;
        c->exps = c->useful_pv_macs / (uint64_t)d_k;
        return PSA_OK;
    }
    // bf16: walk the CTA list and each CTA's block list exactly as the kernels do.  (Where the kernel hands the last
    // pairs of a launch out as single row tiles, split_point in psa_sched.h, those are the same row tiles with the
    // same block lists taken one at a time: the census does not depend on the grouping.)
    const int T = row_tiles(n);
    // (a head size below the 64, 128 or 256 columns of a tile is zero-padded by the loads; a block counts at that width, also where
    // the products leave steps of zeros out)
    const uint64_t block_macs = (uint64_t)TILE * TILE * (d_k <= 64 ? 64 : (d_k <= 128 ? 128 : 256));
    uint64_t qk_blocks = 0, pv_blocks = 0, exps = 0;
    const int P = ctas_per_head(n);
    for (int cta = 0; cta < P; ++cta) {  // every head has the same list
        const CtaWork w = cta_work(cta, n, scheme == PSA_MASKED, 1, 1);
        for (int t = 0; t < w.ntiles; ++t) {
            const int I = w.tile0 + t, kv = kv_tiles(I, T, scheme);
            pv_blocks += kv;
            if (scheme != PSA_SYMMETRIC) qk_blocks += kv;
            exps += (uint64_t)kv * TILE * TILE;      // every weight of an issued block is exponentiated
        }
    }
    if (scheme == PSA_SYMMETRIC) {
        for (int t = 0; t < sym_pairs(T); ++t) {
            int I, J;
            sym_pair(t, &I, &J);
            if (J <= I) ++qk_blocks;
        }
    }
    c->qk_macs = bh * qk_blocks * block_macs;
    c->pv_macs = bh * pv_blocks * block_macs;
    c->exps = bh * exps;
    return PSA_OK;
}

int psa_last_issued(void* stream, psa_counts* c) {
    if (!c) return PSA_ERR_NULL;
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    if (!cx.last_dc) return PSA_ERR_NULL;
    DeviceCounters h;
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e == cudaSuccess) e = cudaMemcpy(&h, cx.last_dc, sizeof(h), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) { set_cuda_error(e, "psa_last_issued"); return PSA_ERR_CUDA; }
    *c = cx.last_useful;
    c->proj_macs = h.proj_macs;
    c->qk_macs = h.qk_macs;
    c->pv_macs = h.pv_macs;
    c->exps = h.exps;
    return h.status;
}

int psa_measure_pipe_rates(psa_pipe_rates* r, void* stream_v) {
    g_err_text[0] = 0;
    if (!r) return PSA_ERR_NULL;
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || sms <= 0) { set_cuda_error(e, "psa_measure_pipe_rates"); return PSA_ERR_CUDA; }
    const size_t cyc_bytes = align_up(3 * (size_t)sms * sizeof(unsigned long long), 256);
    char* ws = acquire_ws(cx, COUNTER_BYTES + cyc_bytes + 256);
    if (!ws) return PSA_ERR_WORKSPACE;
    cx.clean_ws = nullptr;
    cx.last_dc = nullptr;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    unsigned long long* cyc = reinterpret_cast<unsigned long long*>(ws + COUNTER_BYTES);
    std::vector<unsigned long long> h(3 * (size_t)sms);
    double best[3] = {0, 0, 0};
    for (int rep = 0; rep < 3; ++rep) {       // the first repetition warms the clocks up; the best is kept
        e = cudaMemsetAsync(cyc, 0, cyc_bytes, stream);
        if (e == cudaSuccess) e = launch_pipe_rates(cyc, reinterpret_cast<float*>(ws + COUNTER_BYTES + cyc_bytes), sms, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e == cudaSuccess) e = cudaMemcpy(h.data(), cyc, h.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) { set_cuda_error(e, "psa_measure_pipe_rates"); return PSA_ERR_CUDA; }
        for (int m = 0; m < 3; ++m) {
            std::vector<unsigned long long> v(h.begin() + (size_t)m * sms, h.begin() + (size_t)(m + 1) * sms);
            std::sort(v.begin(), v.end());
            const double med = (double)v[v.size() / 2];
            if (med > 0 && pipe_results_per_launch_per_sm() / med > best[m]) best[m] = pipe_results_per_launch_per_sm() / med;
        }
    }
    r->ex2_per_clk_per_sm = best[0];
    r->fma_per_clk_per_sm = best[1];
    r->softmax_weights_per_clk_per_sm = best[2];
    r->sm_count = sms;
    return PSA_OK;
}

int psa_selftest_wait_expiry(unsigned limit_us, void* stream_v) {
    g_err_text[0] = 0;
    if (limit_us == 0 || limit_us > 100000u) return PSA_ERR_SHAPE;     // at most 0.1 s (1.6 s for the slowest waiter)
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    char* ws = acquire_ws(cx, COUNTER_BYTES);
    if (!ws) return PSA_ERR_WORKSPACE;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_v);
    cudaError_t e = cudaMemsetAsync(ws, 0, COUNTER_BLOCK_BYTES, stream);
    if (e == cudaSuccess) e = launch_wait_expiry(reinterpret_cast<DeviceCounters*>(ws), limit_us, stream);
    if (e != cudaSuccess) { set_cuda_error(e, "psa_selftest_wait_expiry"); return PSA_ERR_CUDA; }
    cx.clean_ws = nullptr;
    cx.last_dc = reinterpret_cast<DeviceCounters*>(ws);
    memset(&cx.last_useful, 0, sizeof(psa_counts));
    return PSA_OK;
}

int psa_last_rescales(void* stream, uint64_t* rescales) {
    if (!rescales) return PSA_ERR_NULL;
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    if (!cx.last_dc) return PSA_ERR_NULL;
    DeviceCounters h;
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e == cudaSuccess) e = cudaMemcpy(&h, cx.last_dc, sizeof(h), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) { set_cuda_error(e, "psa_last_rescales"); return PSA_ERR_CUDA; }
    *rescales = h.rescales;
    return PSA_OK;
}

size_t psa_workspace_bytes(int batch, int heads, int n, int d_model, int d_k, int scheme, int dtype,
                           int with_host_staging) {
    const bool with_proj = d_model > 0;
    if (check_shape(batch, heads, n, d_model, d_k, scheme, dtype, with_proj) != PSA_OK) return 0;
    return ws_layout(call_shape(batch, heads, n, d_model, d_k, scheme, dtype, with_proj, with_host_staging != 0 && with_proj)).total;
}

int psa_set_workspace(void* dev_ptr, size_t bytes) {
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    if (dev_ptr && (reinterpret_cast<uintptr_t>(dev_ptr) & 255u)) return PSA_ERR_ALIGN;
    cx.user_ws = dev_ptr;
    cx.user_bytes = dev_ptr ? bytes : 0;
    cx.last_dc = nullptr;
    cx.clean_ws = nullptr;
    return PSA_OK;
}

int psa_profile_begin(int max_calls) {
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    for (cudaEvent_t e : cx.prof_events) cudaEventDestroy(e);
    cx.prof_events.clear();
    cx.prof_calls = 0;
    cx.prof_max = 0;
    if (max_calls <= 0 || max_calls > 100000) return PSA_ERR_SHAPE;
    cx.prof_events.resize(3 * (size_t)max_calls);
    for (size_t i = 0; i < cx.prof_events.size(); ++i) {
        cudaError_t e = cudaEventCreate(&cx.prof_events[i]);
        if (e != cudaSuccess) {
            set_cuda_error(e, "cudaEventCreate");
            for (size_t k = 0; k < i; ++k) cudaEventDestroy(cx.prof_events[k]);
            cx.prof_events.clear();
            return PSA_ERR_CUDA;
        }
    }
    cx.prof_max = max_calls;
    return PSA_OK;
}

int psa_profile_end(float* proj_ms_sum, float* attn_ms_sum, int* calls) {
    Context* cp = current_ctx();
    if (!cp) return PSA_ERR_CUDA;
    Context& cx = *cp;
    std::lock_guard<std::mutex> lock(cx.mu);
    float p = 0.f, a = 0.f;
    int rc = PSA_OK;
    for (int c = 0; c < cx.prof_calls; ++c) {
        cudaEvent_t* ev = &cx.prof_events[3 * c];
        float t0 = 0.f, t1 = 0.f;
        cudaError_t e = cudaEventSynchronize(ev[2]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t0, ev[0], ev[1]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t1, ev[1], ev[2]);
        if (e != cudaSuccess) { set_cuda_error(e, "psa_profile_end"); rc = PSA_ERR_CUDA; break; }
        p += t0; a += t1;
    }
    if (proj_ms_sum) *proj_ms_sum = p;
    if (attn_ms_sum) *attn_ms_sum = a;
    if (calls) *calls = cx.prof_calls;
    for (cudaEvent_t e : cx.prof_events) cudaEventDestroy(e);
    cx.prof_events.clear();
    cx.prof_calls = 0;
    cx.prof_max = 0;
    return rc;
}

const char* psa_status_string(int status) {
    switch (status) {
        case PSA_OK: return "ok";
        case PSA_ERR_NULL: return "a required pointer is NULL";
        case PSA_ERR_SHAPE: return "invalid size";
        case PSA_ERR_UNSUPPORTED: return "shape or number type not supported by this path";
        case PSA_ERR_ALIGN: return "pointer not sufficiently aligned";
        case PSA_ERR_SCHEME_ARGS: return "unknown scheme, or operands inconsistent with the scheme";
        case PSA_ERR_WORKSPACE: return "workspace unavailable";
        case PSA_ERR_CUDA: return "CUDA call failed";
        case PSA_ERR_TIMEOUT: return "a bounded device-side wait expired";
        case PSA_ERR_NUMERIC: return "numeric failure";
        default: return "unknown status";
    }
}

const char* psa_last_cuda_error(void) { return g_err_text; }

}  // extern "C"
