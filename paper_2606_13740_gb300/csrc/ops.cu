// Single-kernel entry points (include/dllm_ops.h) for kernel-level tests.
#include "../../include/dllm.h"
#include "../../include/dllm_ops.h"
#include "internal.h"

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

using namespace dllm;

extern "C" const char* dllm_last_error(const dllm_ctx* ctx);
void dllm_set_noctx_error(const char* msg);

namespace {

int op_fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    dllm_set_noctx_error(buf);
    return code;
}

int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return n;
}

// The scratch of the projection and LM-head calls is kept from one call for the next, so that a
// call does not pay for cudaMalloc and cudaFree (about 250 us for the 40 MB of split partials of a
// 1024-token projection, beside 150 us on the GPU).  A call takes a kept buffer for itself alone
// and puts it back once it has waited for its kernels, so calls on several streams and from
// several threads never share one.  At most kKeepBytes stay kept for a context.  The buffers are
// plain cudaMalloc memory of their context and end with it (cudaDeviceReset): a buffer is found
// again only under its context's id, which the process never gives out twice.
constexpr size_t kKeepBytes = size_t(64) << 20;

struct KeptBuf {
    unsigned long long ctx;
    void* p;
    size_t bytes;
    KeptBuf* next;
};
std::mutex kept_mu;
KeptBuf* kept = nullptr;  // under kept_mu

// The id of the current context (which the caller has made by an earlier call to the runtime).
bool current_context(unsigned long long* id) {
    typedef CUresult (*GetIdFn)(CUcontext, unsigned long long*);
    static const GetIdFn get_id = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &q);
        return reinterpret_cast<GetIdFn>(e == cudaSuccess && q == cudaDriverEntryPointSuccess ? fn : nullptr);
    }();
    return get_id && get_id(nullptr, id) == CUDA_SUCCESS;
}

// Frees a list of buffers of the current context.
void free_bufs(KeptBuf* b) {
    while (b) {
        KeptBuf* next = b->next;
        cudaFree(b->p);
        delete b;
        b = next;
    }
}

// Takes the smallest kept buffers of a context off the list until the others hold `bytes` at most.
KeptBuf* drop_past(unsigned long long ctx, size_t bytes) {  // under kept_mu
    KeptBuf* out = nullptr;
    for (;;) {
        size_t sum = 0;
        KeptBuf** least = nullptr;
        for (KeptBuf** e = &kept; *e; e = &(*e)->next) {
            if ((*e)->ctx != ctx) continue;
            sum += (*e)->bytes;
            if (!least || (*e)->bytes < (*least)->bytes) least = e;
        }
        if (sum <= bytes) return out;
        KeptBuf* b = *least;
        *least = b->next;
        b->next = out;
        out = b;
    }
}

}  // namespace

bool dllm::free_kept_scratch() {
    unsigned long long ctx = 0;
    if (!current_context(&ctx)) return false;
    KeptBuf* out;
    {
        std::lock_guard<std::mutex> lock(kept_mu);
        out = drop_past(ctx, 0);
    }
    const bool any = out != nullptr;
    free_bufs(out);
    return any;
}

namespace {

// A buffer of at least `bytes`: the smallest kept one that does, else a new one (where memory is
// short, in the place of the kept ones); null: no memory.
KeptBuf* take_buf(size_t bytes) {
    unsigned long long ctx = 0;
    if (!current_context(&ctx)) return nullptr;
    {
        std::lock_guard<std::mutex> lock(kept_mu);
        KeptBuf** best = nullptr;
        for (KeptBuf** e = &kept; *e; e = &(*e)->next)
            if ((*e)->ctx == ctx && (*e)->bytes >= bytes && (!best || (*e)->bytes < (*best)->bytes)) best = e;
        if (best) {
            KeptBuf* b = *best;
            *best = b->next;
            b->next = nullptr;
            return b;
        }
    }
    KeptBuf* b = new (std::nothrow) KeptBuf{ctx, nullptr, bytes, nullptr};
    if (!b) return nullptr;
    if (cudaMalloc(&b->p, bytes) == cudaSuccess) return b;
    cudaGetLastError();
    if (free_kept_scratch() && cudaMalloc(&b->p, bytes) == cudaSuccess) return b;
    cudaGetLastError();
    delete b;
    return nullptr;
}

// Keeps a buffer that no work uses any more, smaller ones dropped where that is too much.
void keep_buf(KeptBuf* b) {
    KeptBuf* out = b;
    if (b->bytes <= kKeepBytes) {
        std::lock_guard<std::mutex> lock(kept_mu);
        out = drop_past(b->ctx, kKeepBytes - b->bytes);
        b->next = kept;
        kept = b;
    }
    free_bufs(out);
}

// One call's scratch, carved from one buffer: zeroed pieces first, then the others.
struct OpScratch {
    KeptBuf* buf = nullptr;
    size_t used = 0;
    bool idle = false;  // the call's work on it is done
    ~OpScratch() {
        if (!buf) return;
        if (idle) keep_buf(buf);
        else free_bufs(buf);
    }
    static size_t rounded(size_t bytes) { return (bytes + 255) / 256 * 256; }
    bool alloc(size_t bytes, size_t zero_bytes, cudaStream_t st) {
        // The calls synchronise, so they are refused, before anything is launched or captured, on a
        // capturing stream and where another stream's capture forbids this thread such calls (the
        // query is one of those).
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
        const cudaError_t query = cudaStreamQuery(st);
        if (query != cudaSuccess && query != cudaErrorNotReady) return false;
        buf = take_buf(bytes);
        return buf && cudaMemsetAsync(buf->p, 0, zero_bytes, st) == cudaSuccess;
    }
    template <typename T>
    T* take(size_t bytes) {
        T* q = reinterpret_cast<T*>(static_cast<uint8_t*>(buf->p) + used);
        used += rounded(bytes);
        return q;
    }
};

// Device scratch owned by one op call.
struct DevBuf {
    void* p = nullptr;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
    bool alloc(size_t bytes) { return cudaMalloc(&p, bytes ? bytes : 16) == cudaSuccess; }
};

// Waits for a call's kernels and reports; buf: its scratch, of which status_dev is a part.
int finish(cudaStream_t st, int* status_dev = nullptr, OpScratch* buf = nullptr) {
    int s = 0;
    cudaError_t e = status_dev ? cudaMemcpyAsync(&s, status_dev, 4, cudaMemcpyDeviceToHost, st) : cudaSuccess;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (buf) buf->idle = e == cudaSuccess;
    if (e != cudaSuccess) return op_fail(DLLM_ECUDA, "%s", cudaGetErrorString(e));
    if (s & kStatusTimeout) return op_fail(DLLM_ETIMEOUT, "bounded device wait ran out");
    if (s) return op_fail(DLLM_ECUDA, "device status %d", s);
    return DLLM_OK;
}

}  // namespace

extern "C" {

static int gemm_impl(const void* W, const void* X, float* D, int M, int N, int K, int grid, int reps, float* ms,
                     void* stream, unsigned long long* trace_host = nullptr, int* grid_out = nullptr, int flags = 0) {
    if (!W || !X || !D || M < 1 || N < 1 || K < 1 || (K * 2) % 16 || reps < 1)
        return op_fail(DLLM_EINVAL, "bad gemm arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int sms = sm_count();
    if (sms <= 0) return op_fail(DLLM_ECUDA, "no CUDA device");
    if (gemm_init_attrs() != cudaSuccess) return op_fail(DLLM_ECUDA, "attribute setup failed");
    // a grid that the caller chose is kept
    GemmPlan p = gemm_plan(M, N, K, (grid > 0 && grid < sms) ? grid : sms, EPI_F32, grid <= 0 && gemm_small(M, N, K, sms));
    p.pdl = false;  // the operands come from the caller's kernels
    CUtensorMap tw, tx;
    if (!make_tmap_bf16(&tw, W, M, K, 128) || !make_tmap_bf16(&tx, X, N, K, p.ntile))
        return op_fail(DLLM_EINVAL, "tensor map encode failed (alignment?)");
    const size_t pf = gemm_partial_floats(p);
    const int cl = p.m_tiles * p.n_tiles * 32;
    const size_t cnt_bytes = static_cast<size_t>(cl) * 4, zero = OpScratch::rounded(16) + OpScratch::rounded(cnt_bytes);
    OpScratch buf;
    if (!buf.alloc(zero + pf * 4, zero, st)) return op_fail(DLLM_ENOMEM, "scratch allocation failed");
    int* status = buf.take<int>(16);
    int* cnt = buf.take<int>(cnt_bytes);
    Scratch scr{buf.take<float>(pf * 4), cnt, pf, cl};
    EpiArgs ep{};
    ep.out = D;
    ep.ld_out = M;
    DevBuf tr;
    if (trace_host) {
        if (!tr.alloc(static_cast<size_t>(p.grid) * 16 * 8)) return op_fail(DLLM_ENOMEM, "trace allocation failed");
        ep.trace = static_cast<unsigned long long*>(tr.p);
    }
    if (grid_out) *grid_out = p.grid;
    if (flags & 4) {
        // the bounded-wait test: one launch whose operand producer waits for a word nobody
        // writes (the zeroed third int of the status allocation; the launch's tag is 1)
        cudaError_t e = gemm_launch(EPI_F32, p, tw, tx, ep, scr, status, st, status + 2);
        if (e != cudaSuccess) return op_fail(DLLM_ECUDA, "gemm launch: %s", cudaGetErrorString(e));
        return finish(st, status, &buf);
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ms && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
        return op_fail(DLLM_ECUDA, "event creation failed");
    cudaError_t e = cudaSuccess;
    if (ms) {
        // one untimed launch first (instruction and descriptor caches)
        e = gemm_launch(EPI_F32, p, tw, tx, ep, scr, status, st);
        if (e == cudaSuccess) e = cudaEventRecord(e0, st);
        // flags bit 0: the timed launches form a programmatic-dependent-launch chain (each one
        // only follows this library's own GEMM, which writes neither operand)
        p.pdl = (flags & 1) != 0;
    }
    for (int r = 0; r < reps && e == cudaSuccess; ++r)
        e = gemm_launch(EPI_F32, p, tw, tx, ep, scr, status, st);
    if (ms && e == cudaSuccess) e = cudaEventRecord(e1, st);
    int rc = DLLM_OK;
    if (e != cudaSuccess) rc = op_fail(DLLM_ECUDA, "gemm launch: %s", cudaGetErrorString(e));
    if (rc == DLLM_OK) rc = finish(st, status, &buf);
    if (rc == DLLM_OK && ms) {
        float t = 0.0f;
        cudaEventElapsedTime(&t, e0, e1);
        *ms = t / reps;
    }
    if (rc == DLLM_OK && trace_host &&
        cudaMemcpy(trace_host, tr.p, static_cast<size_t>(p.grid) * 16 * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = op_fail(DLLM_ECUDA, "trace copy failed");
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return rc;
}

int dllm_op_gemm(const void* W, const void* X, float* D, int M, int N, int K, int grid, void* stream) {
    return gemm_impl(W, X, D, M, N, K, grid, 1, nullptr, stream);
}

int dllm_op_gemm_timed(const void* W, const void* X, float* D, int M, int N, int K, int grid, int reps, int flags,
                       float* ms_per_launch, void* stream) {
    if (!ms_per_launch) return op_fail(DLLM_EINVAL, "null output");
    set_stream_smem(!(flags & 2));
    int rc = gemm_impl(W, X, D, M, N, K, grid, reps, ms_per_launch, stream, nullptr, nullptr, flags);
    set_stream_smem(true);
    return rc;
}

int dllm_op_gemm_trace(const void* W, const void* X, float* D, int M, int N, int K, int grid, int reps,
                       float* ms_per_launch, unsigned long long* trace, int* grid_used, void* stream) {
    if (!ms_per_launch || !trace || !grid_used) return op_fail(DLLM_EINVAL, "null output");
    return gemm_impl(W, X, D, M, N, K, grid, reps, ms_per_launch, stream, trace, grid_used);
}

int dllm_op_attention(const void* q, const void* kc, const void* vc, const int32_t* kv_len, void* out, int B, int T,
                      int H, int Hkv, int hd, int cap, int max_kv_len, void* stream) {
    if (!q || !kc || !vc || !kv_len || !out || B < 1 || T < 1 || H < 1 || Hkv < 1 || H % Hkv ||
        (hd != 64 && hd != 128) || max_kv_len < 0 || max_kv_len + T > cap)
        return op_fail(DLLM_EINVAL, "bad attention arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int sms = sm_count();
    if (sms <= 0) return op_fail(DLLM_ECUDA, "no CUDA device");
    if (attn_init_attrs() != cudaSuccess) return op_fail(DLLM_ECUDA, "attribute setup failed");
    AttnPlan a = attn_plan(B, T, H, Hkv, hd, max_kv_len + T, sms);
    cudaError_t e = launch_attention(static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(kc),
                                     static_cast<const __nv_bfloat16*>(vc), kv_len, static_cast<__nv_bfloat16*>(out),
                                     B, T, H, Hkv, hd, cap, a, st, false);
    if (e != cudaSuccess) return op_fail(DLLM_ECUDA, "attention launch: %s", cudaGetErrorString(e));
    return finish(st);
}

int dllm_op_lmhead(const void* W, const void* X, const int32_t* cur, int32_t* x0, float* conf, float* tokconf,
                   float* logits, int V, int N, int d, int mask_id, void* stream) {
    if (!W || !X || !cur || !x0 || !conf || !tokconf || V < 2 || N < 1 || d < 8 || (d * 2) % 16 || mask_id < 0 ||
        mask_id >= V)
        return op_fail(DLLM_EINVAL, "bad lmhead arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int sms = sm_count();
    if (sms <= 0) return op_fail(DLLM_ECUDA, "no CUDA device");
    if (gemm_init_attrs() != cudaSuccess) return op_fail(DLLM_ECUDA, "attribute setup failed");
    GemmPlan p = gemm_plan(V, N, d, sms, EPI_LMHEAD, gemm_small(V, N, d, sms));
    p.pdl = false;
    CUtensorMap tw, tx;
    if (!make_tmap_bf16(&tw, W, V, d, 128) || !make_tmap_bf16(&tx, X, N, d, p.ntile))
        return op_fail(DLLM_EINVAL, "tensor map encode failed (alignment?)");
    const size_t pf = gemm_partial_floats(p);
    const int cl = p.m_tiles * p.n_tiles * 32;
    const size_t cnt_bytes = static_cast<size_t>(cl) * 4, zc_bytes = static_cast<size_t>(N) * 4;
    const size_t lmp_bytes = static_cast<size_t>(p.m_tiles) * N * 3 * 4;
    const size_t zero = OpScratch::rounded(16) + OpScratch::rounded(cnt_bytes) + OpScratch::rounded(zc_bytes);
    OpScratch buf;
    if (!buf.alloc(zero + OpScratch::rounded(lmp_bytes) + pf * 4, zero, st))
        return op_fail(DLLM_ENOMEM, "scratch allocation failed");
    int* status = buf.take<int>(16);
    int* cnt = buf.take<int>(cnt_bytes);
    float* zc = buf.take<float>(zc_bytes);
    float* lmp = buf.take<float>(lmp_bytes);
    Scratch scr{buf.take<float>(pf * 4), cnt, pf, cl};
    EpiArgs ep{};
    ep.lm_part = lmp;
    ep.zcur = zc;
    ep.cur_tok = cur;
    ep.logits = logits;
    ep.V = V;
    ep.mask_id = mask_id;
    cudaError_t e = gemm_launch(EPI_LMHEAD, p, tw, tx, ep, scr, status, st);
    if (e == cudaSuccess)
        e = launch_lmhead_reduce(lmp, zc, cur, p.m_tiles, N, mask_id, x0, conf, tokconf, st, false);
    if (e != cudaSuccess) return op_fail(DLLM_ECUDA, "lmhead launch: %s", cudaGetErrorString(e));
    return finish(st, status, &buf);
}

void dllm_op_release_scratch(void) { free_kept_scratch(); }

int dllm_op_commit(int32_t* tok, uint8_t* status, int n_pos, int w0, int T, int c0, int c1, int step,
                   const int32_t* x0, const float* conf, const float* tokconf, int steps_per_block,
                   float theta_remask, float theta_stable, int remask_max, int spec_blocks, int use_prefix_cache,
                   int block_len, int mask_id, int commit_mode, float theta_visible, int* out6) {
    if (!tok || !status || !x0 || !conf || !tokconf || n_pos < 1 || T < 1 || w0 < 0 || w0 + T > n_pos || c0 < w0 ||
        c1 > w0 + T || c0 > c1 || c1 - c0 > kMaxBlock || steps_per_block < 1 || block_len < 1 ||
        (commit_mode != DLLM_COMMIT_SCHEDULE && commit_mode != DLLM_COMMIT_THRESHOLD))
        return op_fail(DLLM_EINVAL, "bad commit arguments");
    if (!use_prefix_cache && w0 != 0) return op_fail(DLLM_EINVAL, "without the prefix cache the window starts at 0");
    DevBuf dtok, dst, dx0, dconf, dtc, dkv, dplan, douts;
    if (!dtok.alloc(static_cast<size_t>(n_pos) * 4) || !dst.alloc(n_pos) || !dx0.alloc(static_cast<size_t>(T) * 4) ||
        !dconf.alloc(static_cast<size_t>(T) * 4) || !dtc.alloc(static_cast<size_t>(T) * 4) || !dkv.alloc(4) ||
        !dplan.alloc(16) || !douts.alloc(32))
        return op_fail(DLLM_ENOMEM, "allocation failed");
    int plan[4] = {c0, c1, step, 0};
    bool ok = cudaMemcpy(dtok.p, tok, static_cast<size_t>(n_pos) * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dst.p, status, n_pos, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dx0.p, x0, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dconf.p, conf, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dtc.p, tokconf, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dkv.p, &w0, 4, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(dplan.p, plan, 16, cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) return op_fail(DLLM_ECUDA, "copy in failed");
    CommitArgs a{};
    a.tok = static_cast<int*>(dtok.p);
    a.st = static_cast<uint8_t*>(dst.p);
    a.ld = n_pos;
    a.seq_kv = static_cast<int*>(dkv.p);
    a.plan = static_cast<int*>(dplan.p);
    a.x0 = static_cast<int*>(dx0.p);
    a.conf = static_cast<float*>(dconf.p);
    a.tokconf = static_cast<float*>(dtc.p);
    a.outs = static_cast<int*>(douts.p);
    a.B = 1;
    a.T = T;
    a.mask_id = mask_id;
    a.use_cache = use_prefix_cache;
    a.S = steps_per_block;
    a.remask_max = remask_max;
    a.spec_blocks = spec_blocks;
    a.block_len = block_len;
    a.theta_remask = theta_remask;
    a.theta_stable = theta_stable;
    a.commit_mode = commit_mode;
    a.theta_visible = theta_visible;
    a.Tq = T;  // window rows only (no sparse cache refresh rows)
    cudaError_t e = launch_commit(a, nullptr, false);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return op_fail(DLLM_ECUDA, "commit: %s", cudaGetErrorString(e));
    int outs[8];
    ok = cudaMemcpy(tok, dtok.p, static_cast<size_t>(n_pos) * 4, cudaMemcpyDeviceToHost) == cudaSuccess &&
         cudaMemcpy(status, dst.p, n_pos, cudaMemcpyDeviceToHost) == cudaSuccess &&
         cudaMemcpy(outs, douts.p, 32, cudaMemcpyDeviceToHost) == cudaSuccess;
    if (!ok) return op_fail(DLLM_ECUDA, "copy out failed");
    if (out6) memcpy(out6, outs, 6 * sizeof(int));
    return DLLM_OK;
}

}  // extern "C"
