// C ABI of the batched Dilithium engine (declarations and contracts in
// include/dil.h).  Host-side argument checking, the device workspace owned by a
// context, batch chunking to the workspace budget, and the host-buffer forms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include <nvtx3/nvToolsExt.h>

#include "../../include/dil.h"
#include "dil_launch.h"

struct dil_ctx {
    int device = 0;
    size_t budget = 0;
    void *ws = nullptr;       // device scratch
    size_t ws_bytes = 0;
    int max_iter = 0;         // 0 = nonce cap
    // launch shape per operation (keygen / sign / verify) and level (2 / 3 / 5)
    // as set by dil_set_tuning; 0: not set
    int warps[3][3] = {};   // warps per CTA
    int wpt[3][3] = {};     // warps per task
    // host-form staging (device memory)
    void *stage = nullptr;
    size_t stage_bytes = 0;
    // persistent Sign: workspace, tuning and the cached captured launch
    void *pws = nullptr;
    size_t pws_bytes = 0;
    dil::PersistTuning ptune;
    bool ptune_set = false;   // by dil_set_persistent_tuning
    cudaStream_t cap_stream = nullptr;
    cudaStream_t cancel_stream = nullptr;   // carries the cancel word's copy
    cudaGraphExec_t gexec = nullptr;
    dil::PersistJobs gjobs{};
    dil::PersistTuning gtune;
    bool gwish = false;       // it was to run in rounds
    int gmax_iter = -1;
    int spin_limit = 0;       // polls per bounded device wait (0 = PERSIST_SPIN_LIMIT); tests lower it
    int gspin_limit = -1;
    void *gws = nullptr;
    size_t alloc_limit = 0;   // larger persistent workspaces count as refused (0: none); a test sets it
    // host-form pipeline: extra streams and the fork / join events
    cudaStream_t aux[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::mutex mu;
};

namespace {

constexpr size_t POLY_BYTES = 256 * sizeof(int32_t);

// NVTX range over one API call (a no-op unless a profiler is attached), so
// traces show which entry point issued which launches.
struct TraceRange {
    explicit TraceRange(const char *name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange &) = delete;
    TraceRange &operator=(const TraceRange &) = delete;
};

bool level_ok(int level) { return level == 2 || level == 3 || level == 5; }
int lidx(int level) { return level == 2 ? 0 : level == 3 ? 1 : 2; }

int cuda_fail(cudaError_t e) { return e == cudaErrorMemoryAllocation ? DIL_ENOMEM : DIL_ECUDA; }

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

// Ensures at least `bytes` of workspace; returns DIL_OK or an error.
int ensure_ws(dil_ctx *c, size_t bytes) {
    if (bytes <= c->ws_bytes) return DIL_OK;
    if (bytes > c->budget) return DIL_ENOMEM;
    if (c->ws) {
        cudaDeviceSynchronize();
        cudaFree(c->ws);
        c->ws = nullptr;
        c->ws_bytes = 0;
    }
    cudaError_t e = cudaMalloc(&c->ws, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        c->ws = nullptr;
        return DIL_ENOMEM;
    }
    c->ws_bytes = bytes;
    return DIL_OK;
}

// Largest number of tasks per launch whose scratch (`per` bytes each) fits the budget.
size_t chunk_tasks(const dil_ctx *c, size_t per, size_t n) {
    return std::min<size_t>(n, std::min<size_t>(c->budget / per, (size_t)1 << 30));
}
size_t chunk_tasks(const dil_ctx *c, int op, int level, size_t n) {
    return chunk_tasks(c, dil::scratch_polys(op, level) * POLY_BYTES, n);
}

// Tasks of a part when a batch runs in parts on ns streams, each with a part's
// scratch; one stream when the budget does not hold ns tasks' scratch.
size_t part_tasks(const dil_ctx *c, size_t n, size_t per, size_t &ns) {
    if (c->budget < ns * per) ns = 1;
    return std::min((n + ns - 1) / ns, chunk_tasks(c, ns * per, n));
}

// Launch shape of one call.  The fused forms run when the caller asked for two
// or four warps per task (a task of theirs needs at least the scratch of the batch
// form's; Sign's rounds need a little more, sign_fused).
struct Shape {
    bool fused;
    int warps, p;
};

Shape shape_of(const dil_ctx *c, int op, int level) {
    const int w = c->warps[op][lidx(level)], p = c->wpt[op][lidx(level)];
    return {p > 1, w, p};
}

// The fused kernels' launch shape where a caller set none.
int fused_warps(const dil_ctx *c, int op, int level) { const int w = c->warps[op][lidx(level)]; return w ? w : 8; }
int fused_wpt(const dil_ctx *c, int op, int level) { const int p = c->wpt[op][lidx(level)]; return p ? p : 2; }

// Tasks and slots of one launch of Sign in rounds within `budget` bytes; tasks
// is 0 when not even one fits.
struct RoundSize {
    size_t tasks, slots;
};

RoundSize round_size(int level, int src, size_t n, size_t budget, int parts = 1) {
    size_t m = std::min<size_t>(n, (size_t)1 << 24);
    while (m > 0) {
        const size_t wish = dil::sign_batch_slots(level, (int)m, parts), least = dil::sign_batch_min_slots(level, (int)m);
        if (dil::sign_batch_bytes(level, src, m, wish) <= budget) return {m, wish};
        const size_t need = dil::sign_batch_bytes(level, src, m, least);
        if (need <= budget) return {m, least};
        m = std::min(m - 1, (size_t)((double)m * budget / need));
    }
    return {0, 0};
}

// The Sign form of a call: the fused kernel as for the other operations (shape_of),
// and where the budget holds the scratch of one of its tasks but no round.
bool sign_fused(const dil_ctx *c, int level, int src) {
    return c->wpt[1][lidx(level)] > 1 || round_size(level, src, 1, c->budget).tasks == 0;
}

// Streams a KeyGen batch is spread over: one half's arithmetic and tr beside the
// other's sampling.  On one and two streams 5,000 and 10,000 Dilithium2 keys take
// 271, 454 and 265, 437 us, 10,000 and 16,000 Dilithium3 756, 1114 and 728, 1111;
// but 3,000 and 4,000 Dilithium2 192, 225 and 220, 253, 2,048 and 6,000 Dilithium3
// 234, 484 and 411, 530, 6,000, 10,000 and 20,000 Dilithium5 759, 1209, 2269 and 827,
// 1196, 2311.
size_t keygen_parts(int level, size_t n) { return n >= (level == 2 ? 5000u : 9000u) && level != 5 ? 2 : 1; }

cudaError_t keygen_chunk(const Shape &sh, int level, int m, const uint8_t *seeds, uint8_t *pk, uint8_t *sk,
                         int32_t *scratch, cudaStream_t s) {
    return sh.fused ? dil::launch_keygen(level, m, seeds, pk, sk, scratch, sh.warps, sh.p, s)
                    : dil::launch_keygen_batch(level, m, seeds, pk, sk, scratch, s);
}

size_t verify_task_bytes(int level, int src) {
    return dil::verify_batch_polys(level, src) * POLY_BYTES + dil::VERIFY_AUX_BYTES;
}

constexpr size_t PIPE_MIN_TASKS = 2048;   // smaller batches run as one chunk
constexpr size_t PIPE_STREAMS = 4;

// The context's first `streams` own streams and the fork / join events (made when
// a call first needs them: a stream costs a context's first Verify 7 us).
int ensure_aux(dil_ctx *c, size_t streams) {
    bool ok = true;
    for (size_t i = 0; i < streams && ok; ++i)
        if (!c->aux[i]) ok = cudaStreamCreateWithFlags(&c->aux[i], cudaStreamNonBlocking) == cudaSuccess;
    for (cudaEvent_t *e : {&c->ev_fork, &c->ev_join})
        if (ok && !*e) ok = cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok ? DIL_OK : DIL_ECUDA;
}

// Runs chunk(c0, c1, stream, scratch) over n tasks, `per` at a time, on ns streams
// (the caller's and the context's others) that start after what is on the
// caller's and that it waits for.  `region` is a chunk's kernel scratch in bytes.
template <class Chunk>
int run_streams(dil_ctx *c, size_t n, size_t per, size_t region, size_t ns, cudaStream_t s0, Chunk chunk) {
    if (per == 0) return DIL_ENOMEM;
    const size_t k = (n + per - 1) / per;
    ns = std::min(ns, k);
    int rc = ensure_ws(c, ns * region);
    if (!rc && ns > 1) rc = ensure_aux(c, ns - 1);
    if (rc) return rc;
    cudaStream_t st[PIPE_STREAMS] = {s0, c->aux[0], c->aux[1], c->aux[2]};
    if (ns > 1) {
        if (cudaEventRecord(c->ev_fork, s0) != cudaSuccess) return DIL_ECUDA;
        for (size_t j = 1; j < ns; ++j)
            if (cudaStreamWaitEvent(st[j], c->ev_fork, 0) != cudaSuccess) return DIL_ECUDA;
    }
    for (size_t i = 0; i < k && !rc; ++i) {
        const size_t c0 = i * per, c1 = std::min(n, c0 + per);
        int32_t *scratch = (int32_t *)c->ws + (i % ns) * (region / sizeof(int32_t));
        rc = chunk(c0, c1, st[i % ns], scratch);
    }
    for (size_t j = 1; j < ns; ++j)
        if ((cudaEventRecord(c->ev_join, st[j]) != cudaSuccess ||
             cudaStreamWaitEvent(s0, c->ev_join, 0) != cudaSuccess) && !rc)
            rc = DIL_ECUDA;
    return rc;
}

// Streams a Sign batch of n tasks is spread over: the rounds of one part fill
// the gaps of the others' (the hashes' chains, the ends of kernels).
// 10,000 Dilithium2 tasks on 2, 3, 4 streams: 1593, 1546, 1524 us; 10,000
// Dilithium3 2295, 2253, 2233; 3,000 Dilithium2 707, 680, 672.  (Streams of
// falling priority: 1700 and 2460 us for the first two.)
size_t sign_parts(size_t n) { return n >= PIPE_MIN_TASKS ? PIPE_STREAMS : 1; }

// Runs Sign in rounds over the n tasks of `all` (whose per-task pointers are
// those of task 0), in as many launches as the budget asks for.
int run_sign_batch(dil_ctx *c, int level, int src, size_t n, const dil::SignBatch &all, cudaStream_t s) {
    size_t ns = sign_parts(n);
    RoundSize z = round_size(level, src, (n + ns - 1) / ns, c->budget / ns, (int)ns);
    if (z.tasks == 0) z = round_size(level, src, n, c->budget, (int)(ns = 1));
    size_t pkb, skb, sigb;
    dil_sizes(level, &pkb, &skb, &sigb);
    const size_t k = level == 2 ? 4 : level == 3 ? 6 : 8, l = level == 2 ? 4 : level == 3 ? 5 : 7;
    return run_streams(c, n, z.tasks, dil::sign_batch_bytes(level, src, z.tasks, z.slots), ns, s,
                       [&](size_t c0, size_t c1, cudaStream_t st, int32_t *scratch) -> int {
                           dil::SignBatch b = all;
                           b.n = (int)(c1 - c0);
                           b.slots = (int)z.slots;
                           b.parts = (int)ns;
                           b.on_gpu = (int)std::min(n, ns * z.tasks);
                           if (src != dil::SIGN_KEYED) b.sk += skb * c0;
                           if (b.ahat) b.ahat += k * l * 256 * c0;
                           if (b.key_idx) b.key_idx += c0;
                           b.off += c0;
                           b.sig += sigb * c0;
                           if (b.status) b.status += c0;
                           if (b.iters) b.iters += c0;
                           const cudaError_t e = dil::launch_sign_batch(level, src, b, scratch, st);
                           return e == cudaSuccess ? DIL_OK : cuda_fail(e);
                       });
}

// Carves m tasks of a Verify batch out of a workspace of m verify_task_bytes.
void carve_verify(dil::VerifyBatch &b, void *ws, size_t m, size_t polys) {
    uint8_t *aux = static_cast<uint8_t *>(ws) + m * polys * POLY_BYTES;
    b.n = (int)m;
    b.scratch = static_cast<int32_t *>(ws);
    b.mu = reinterpret_cast<uint32_t *>(aux);
    b.tr = reinterpret_cast<uint32_t *>(aux + 64 * m);
    b.next = reinterpret_cast<int *>(aux + 96 * m);
    b.challenge = aux + 128 * m;
}

// Runs Verify's batch form over the n tasks of `all` (whose per-task pointers are
// those of task 0), in as many launches as the budget asks for, with the hashes
// on a stream of their own.  (Parts of a large batch on several streams gain
// nothing that holds: with the hashes between two halves' sampling 10,000
// Dilithium2 tasks take 408 us instead of 416, 10,000 Dilithium5 1264 instead of
// 1202; the hashes before the sampling cost both 5 to 12%.)
int run_verify_batch(dil_ctx *c, int level, int src, size_t n, const dil::VerifyBatch &all, cudaStream_t s) {
    const size_t polys = dil::verify_batch_polys(level, src), per = verify_task_bytes(level, src);
    const size_t tasks = chunk_tasks(c, per, n);
    const int rc = ensure_aux(c, 1);
    if (rc) return rc;
    size_t pkb, skb, sigb;
    dil_sizes(level, &pkb, &skb, &sigb);
    const size_t k = level == 2 ? 4 : level == 3 ? 6 : 8, l = level == 2 ? 4 : level == 3 ? 5 : 7;
    return run_streams(c, n, tasks, tasks * per, 1, s, [&](size_t c0, size_t c1, cudaStream_t st, int32_t *scratch) -> int {
        dil::VerifyBatch b = all;
        carve_verify(b, scratch, c1 - c0, polys);
        if (src != dil::VERIFY_KEYED) b.pk += pkb * c0;
        if (b.ahat) b.ahat += k * l * 256 * c0;
        if (b.key_idx) b.key_idx += c0;
        b.off += c0;
        b.sig += sigb * c0;
        b.ok += c0;
        const cudaError_t e = dil::launch_verify_batch(level, src, b, {c->aux[0], c->ev_fork, c->ev_join}, st);
        return e == cudaSuccess ? DIL_OK : cuda_fail(e);
    });
}

int sign_cap(const dil_ctx *c, int level) {
    const int l = level == 2 ? 4 : level == 3 ? 5 : 7, cap = (65536 - l) / l + 1;
    return (c->max_iter > 0 && c->max_iter < cap) ? c->max_iter : cap;
}

void sizes_of(int level, size_t &pk, size_t &sk, size_t &sig) { dil_sizes(level, &pk, &sk, &sig); }

}  // namespace

extern "C" {

int dil_sizes(int level, size_t *pk_bytes, size_t *sk_bytes, size_t *sig_bytes) {
    size_t pk, sk, sig;
    switch (level) {
        case 2: pk = 1312; sk = 2528; sig = 2420; break;
        case 3: pk = 1952; sk = 4000; sig = 3293; break;
        case 5: pk = 2592; sk = 4864; sig = 4595; break;
        default: return DIL_EINVAL;
    }
    if (pk_bytes) *pk_bytes = pk;
    if (sk_bytes) *sk_bytes = sk;
    if (sig_bytes) *sig_bytes = sig;
    return DIL_OK;
}

const char *dil_status_string(int status) {
    switch (status) {
        case DIL_OK: return "ok";
        case DIL_EINVAL: return "invalid argument";
        case DIL_ENOMEM: return "out of workspace or device memory";
        case DIL_ECUDA: return "CUDA error";
        case DIL_ETIMEOUT: return "device wait timed out";
        case DIL_EITER: return "sign repetition cap reached";
        case DIL_ECANCELED: return "canceled";
    }
    return "unknown status";
}

int dil_ctx_create(int device, size_t workspace_budget, dil_ctx **out) {
    if (!out) return DIL_EINVAL;
    *out = nullptr;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess) {
        cudaGetLastError();
        return DIL_ECUDA;
    }
    if (device < 0 || device >= count) return DIL_EINVAL;
    dil_ctx *c = new dil_ctx;
    c->device = device;
    c->budget = workspace_budget ? workspace_budget : ((size_t)8 << 30);
    *out = c;
    return DIL_OK;
}

int dil_ctx_destroy(dil_ctx *c) {
    if (!c) return DIL_OK;
    {
        DeviceGuard g(c->device);
        cudaDeviceSynchronize();
        if (c->ws) cudaFree(c->ws);
        if (c->stage) cudaFree(c->stage);
        if (c->pws) cudaFree(c->pws);
        if (c->gexec) cudaGraphExecDestroy(c->gexec);
        if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
        if (c->cancel_stream) cudaStreamDestroy(c->cancel_stream);
        for (cudaStream_t a : c->aux)
            if (a) cudaStreamDestroy(a);
        if (c->ev_fork) cudaEventDestroy(c->ev_fork);
        if (c->ev_join) cudaEventDestroy(c->ev_join);
    }
    delete c;
    return DIL_OK;
}

int dil_set_tuning(dil_ctx *c, int op, int level, int warps_per_cta, int warps_per_task) {
    if (!c || op < 0 || op > 2 || warps_per_cta < 1 || warps_per_cta > 8) return DIL_EINVAL;
    if (level != 0 && !level_ok(level)) return DIL_EINVAL;
    if (warps_per_task != 1 && warps_per_task != 2 && warps_per_task != 4) return DIL_EINVAL;
    if (warps_per_cta % warps_per_task) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    for (int li = 0; li < 3; ++li) {
        if (level && lidx(level) != li) continue;
        c->warps[op][li] = warps_per_cta;
        c->wpt[op][li] = warps_per_task;
    }
    return DIL_OK;
}

int dil_set_max_iter(dil_ctx *c, int max_iter) {
    if (!c || max_iter < 0) return DIL_EINVAL;
    c->max_iter = max_iter;
    return DIL_OK;
}

int dil_keygen(dil_ctx *c, int level, size_t n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, void *stream) {
    TraceRange trace("dil_keygen");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!seeds || !pk || !sk || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const size_t per = dil::scratch_polys(dil::OP_KEYGEN, level) * POLY_BYTES;
    const Shape sh = shape_of(c, 0, level);
    size_t ns = sh.fused ? 1 : keygen_parts(level, n);
    const size_t tasks = part_tasks(c, n, per, ns);
    return run_streams(c, n, tasks, tasks * per, ns, (cudaStream_t)stream,
                       [&](size_t c0, size_t c1, cudaStream_t s, int32_t *scratch) -> int {
                           const cudaError_t e = keygen_chunk(sh, level, (int)(c1 - c0), seeds + 32 * c0, pk + pkb * c0,
                                                              sk + skb * c0, scratch, s);
                           return e == cudaSuccess ? DIL_OK : cuda_fail(e);
                       });
}

int dil_sign_ex(dil_ctx *c, int level, size_t n, const uint8_t *sk, const uint8_t *msg, const uint64_t *msg_off,
                uint8_t *sig, int32_t *task_status, int32_t *iterations, void *stream) {
    TraceRange trace("dil_sign_ex");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!sk || !msg_off || !sig || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const int max_iter = sign_cap(c, level);
    if (!sign_fused(c, level, dil::SIGN_PLAIN)) {
        dil::SignBatch b{};
        b.sk = sk;
        b.msg = msg;
        b.off = msg_off;
        b.sig = sig;
        b.status = task_status;
        b.iters = iterations;
        b.max_iter = max_iter;
        return run_sign_batch(c, level, dil::SIGN_PLAIN, n, b, (cudaStream_t)stream);
    }
    size_t chunk = chunk_tasks(c, dil::OP_SIGN, level, n);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * dil::scratch_polys(dil::OP_SIGN, level) * POLY_BYTES);
    if (rc) return rc;
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        int m = (int)std::min(chunk, n - s0);
        cudaError_t e = dil::launch_sign(level, m, sk + skb * s0, msg, msg_off + s0, sig + sigb * s0,
                                         task_status ? task_status + s0 : nullptr,
                                         iterations ? iterations + s0 : nullptr, (int32_t *)c->ws, max_iter,
                                         fused_warps(c, 1, level), fused_wpt(c, 1, level), (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    return DIL_OK;
}

int dil_sign(dil_ctx *c, int level, size_t n, const uint8_t *sk, const uint8_t *msg, const uint64_t *msg_off,
             uint8_t *sig, int32_t *task_status, void *stream) {
    return dil_sign_ex(c, level, n, sk, msg, msg_off, sig, task_status, nullptr, stream);
}

int dil_verify(dil_ctx *c, int level, size_t n, const uint8_t *pk, const uint8_t *msg, const uint64_t *msg_off,
               const uint8_t *sig, uint8_t *ok, void *stream) {
    TraceRange trace("dil_verify");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!pk || !msg_off || !sig || !ok || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const Shape sh = shape_of(c, 2, level);
    if (!sh.fused) {
        dil::VerifyBatch b{};
        b.pk = pk;
        b.msg = msg;
        b.off = msg_off;
        b.sig = sig;
        b.ok = ok;
        return run_verify_batch(c, level, dil::VERIFY_PLAIN, n, b, (cudaStream_t)stream);
    }
    const size_t per = dil::scratch_polys(dil::OP_VERIFY, level) * POLY_BYTES;
    size_t chunk = chunk_tasks(c, per, n);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * per);
    if (rc) return rc;
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        int m = (int)std::min(chunk, n - s0);
        cudaError_t e = dil::launch_verify(level, m, pk + pkb * s0, msg, msg_off + s0, sig + sigb * s0, ok + s0,
                                           (int32_t *)c->ws, sh.warps, sh.p, (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    return DIL_OK;
}

// ---------------------------------------------------------------- caller-owned A^
namespace {
bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }
size_t ahat_words(int level) {
    const int k = level == 2 ? 4 : level == 3 ? 6 : 8, l = level == 2 ? 4 : level == 3 ? 5 : 7;
    return (size_t)k * l * 256;
}
}  // namespace

int dil_expand_a(dil_ctx *c, int level, size_t n, const uint8_t *rho, size_t rho_stride, uint32_t *ahat,
                 void *stream) {
    TraceRange trace("dil_expand_a");
    if (!c || !level_ok(level) || rho_stride < 32) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!rho || !ahat || !aligned16(ahat) || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    cudaError_t e = dil::launch_expand_a(level, (int)n, rho, rho_stride, reinterpret_cast<int32_t *>(ahat),
                                         (cudaStream_t)stream);
    return e != cudaSuccess ? cuda_fail(e) : DIL_OK;
}

int dil_sign_a(dil_ctx *c, int level, size_t n, const uint8_t *sk, const uint8_t *msg, const uint64_t *msg_off,
               const uint32_t *ahat, uint8_t *sig, int32_t *task_status, int32_t *iterations, void *stream) {
    if (!ahat) return dil_sign_ex(c, level, n, sk, msg, msg_off, sig, task_status, iterations, stream);
    TraceRange trace("dil_sign_a");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!sk || !msg_off || !sig || !aligned16(ahat) || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const int max_iter = sign_cap(c, level);
    if (round_size(level, dil::SIGN_AHAT, 1, c->budget).tasks) {
        dil::SignBatch b{};
        b.sk = sk;
        b.msg = msg;
        b.off = msg_off;
        b.sig = sig;
        b.status = task_status;
        b.iters = iterations;
        b.ahat = reinterpret_cast<const int32_t *>(ahat);
        b.max_iter = max_iter;
        return run_sign_batch(c, level, dil::SIGN_AHAT, n, b, (cudaStream_t)stream);
    }
    // a budget for the fused kernel's scratch of a task, but not for a round's
    const size_t chunk = chunk_tasks(c, dil::OP_SIGN, level, n);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * dil::scratch_polys(dil::OP_SIGN, level) * POLY_BYTES);
    if (rc) return rc;
    const int32_t *a = reinterpret_cast<const int32_t *>(ahat);
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        const int m = (int)std::min(chunk, n - s0);
        cudaError_t e = dil::launch_sign_a(level, m, sk + skb * s0, msg, msg_off + s0, a + ahat_words(level) * s0,
                                           sig + sigb * s0, task_status ? task_status + s0 : nullptr,
                                           iterations ? iterations + s0 : nullptr, (int32_t *)c->ws, max_iter,
                                           fused_warps(c, 1, level), (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    return DIL_OK;
}

int dil_verify_a(dil_ctx *c, int level, size_t n, const uint8_t *pk, const uint8_t *msg, const uint64_t *msg_off,
                 const uint8_t *sig, const uint32_t *ahat, uint8_t *ok, void *stream) {
    if (!ahat) return dil_verify(c, level, n, pk, msg, msg_off, sig, ok, stream);
    TraceRange trace("dil_verify_a");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!pk || !msg_off || !sig || !ok || !aligned16(ahat) || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    dil::VerifyBatch b{};
    b.pk = pk;
    b.msg = msg;
    b.off = msg_off;
    b.sig = sig;
    b.ok = ok;
    b.ahat = reinterpret_cast<const int32_t *>(ahat);
    return run_verify_batch(c, level, dil::VERIFY_AHAT, n, b, (cudaStream_t)stream);
}

// ---------------------------------------------------------------- persistent
int dil_set_persistent_tuning(dil_ctx *c, int warps_per_cta, int warps_per_task, int ctas_per_sm, int chunk,
                              int speculation) {
    if (!c || warps_per_cta < 1 || warps_per_cta > 8 || ctas_per_sm < 0 || chunk < 1 || speculation < 0)
        return DIL_EINVAL;
    if (warps_per_task != 1 && warps_per_task != 2 && warps_per_task != 4) return DIL_EINVAL;
    if (warps_per_cta % warps_per_task) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    c->ptune.warps = warps_per_cta;
    c->ptune.p = warps_per_task;
    c->ptune.ctas_per_sm = ctas_per_sm;
    c->ptune.chunk = chunk;
    c->ptune.spec = speculation;
    c->ptune_set = true;
    return DIL_OK;
}

namespace {
bool same_jobs(const dil::PersistJobs &a, const dil::PersistJobs &b) { return memcmp(&a, &b, sizeof(a)) == 0; }
bool same_tune(const dil::PersistTuning &a, const dil::PersistTuning &b) {
    return a.warps == b.warps && a.p == b.p && a.ctas_per_sm == b.ctas_per_sm && a.chunk == b.chunk &&
           a.spec == b.spec;
}
}  // namespace

namespace {
// A persistent launch in rounds: each job in parts, the parts dealt over the four
// streams; a part's workspace serves one after the other.  At most PART_MOST
// tasks a part: a cancel ends those in flight with their round, and the ones behind
// them leave their work out.
constexpr size_t PART_MOST = 16384;
struct RoundPlan {
    RoundSize size[dil::PERSIST_MAX_JOBS];
    size_t region = 0, bytes = 0;   // a stream's workspace, the launch's (0: does not fit)
};

RoundPlan round_plan(const dil::PersistJobs &J, size_t bytes) {
    RoundPlan p;
    const size_t budget = bytes > dil::PERSIST_HEADER_BYTES ? (bytes - dil::PERSIST_HEADER_BYTES) / PIPE_STREAMS : 0;
    for (int j = 0; j < J.njobs; ++j) {
        const size_t n = J.job[j].n;
        if (n == 0) continue;
        const size_t part = n < PIPE_MIN_TASKS ? n : std::min((n + PIPE_STREAMS - 1) / PIPE_STREAMS, PART_MOST);
        p.size[j] = round_size(J.job[j].level, dil::SIGN_PLAIN, part, budget, PIPE_STREAMS);
        if (p.size[j].tasks == 0) return RoundPlan{};
        p.region = std::max(p.region, dil::sign_batch_bytes(J.job[j].level, dil::SIGN_PLAIN, p.size[j].tasks,
                                                            p.size[j].slots));
    }
    p.bytes = dil::PERSIST_HEADER_BYTES + PIPE_STREAMS * p.region;
    return p;
}

// Ensures `bytes` of persistent workspace; DIL_ENOMEM when the device refuses it
// (the context then holds none).
int ensure_pws(dil_ctx *c, size_t bytes) {
    if (bytes <= c->pws_bytes) return DIL_OK;
    if (c->pws) {
        cudaDeviceSynchronize();
        if (c->gexec) cudaGraphExecDestroy(c->gexec);   // of the old address, which a smaller workspace may get
        c->gexec = nullptr;
        cudaFree(c->pws);
        c->pws = nullptr;
        c->pws_bytes = 0;
    }
    if ((c->alloc_limit && bytes > c->alloc_limit) || cudaMalloc(&c->pws, bytes) != cudaSuccess) {
        cudaGetLastError();
        c->pws = nullptr;
        return DIL_ENOMEM;
    }
    c->pws_bytes = bytes;
    return DIL_OK;
}

// A plan of rounds within `bytes` and its workspace; where the device refuses that
// much, half as much at a time while that is `least` or more.
RoundPlan planned_rounds(dil_ctx *c, const dil::PersistJobs &J, size_t bytes, size_t least) {
    RoundPlan p = round_plan(J, bytes);
    while (p.bytes && ensure_pws(c, p.bytes) != DIL_OK)
        p = p.bytes / 2 < least ? RoundPlan{} : round_plan(J, p.bytes / 2);
    return p;
}

// Enqueues the launch on s and the context's other streams.
cudaError_t launch_rounds(dil_ctx *c, const dil::PersistJobs &J, const RoundPlan &p, cudaStream_t s) {
    cudaStream_t st[PIPE_STREAMS] = {s, c->aux[0], c->aux[1], c->aux[2]};
    cudaError_t e = cudaMemsetAsync(c->pws, 0, dil::PERSIST_HEADER_BYTES, s);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_fork, s);
    for (size_t k = 1; k < PIPE_STREAMS && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(st[k], c->ev_fork, 0);
    size_t turn = 0;
    for (int j = 0; j < J.njobs && e == cudaSuccess; ++j) {
        const dil::PersistJob &x = J.job[j];
        size_t pkb, skb, sigb;
        dil_sizes(x.level, &pkb, &skb, &sigb);
        for (size_t c0 = 0; c0 < (size_t)x.n && e == cudaSuccess; c0 += p.size[j].tasks, ++turn) {
            dil::SignBatch b{};
            b.n = (int)std::min(p.size[j].tasks, x.n - c0);
            b.slots = (int)p.size[j].slots;
            b.parts = PIPE_STREAMS;
            b.on_gpu = J.total;
            b.sk = x.sk + skb * c0;
            b.msg = x.msg;
            b.off = x.off + c0;
            b.sig = x.sig + sigb * c0;
            b.status = x.status ? x.status + c0 : nullptr;
            b.iters = x.iters ? x.iters + c0 : nullptr;
            b.max_iter = sign_cap(c, x.level);
            const size_t k = turn % PIPE_STREAMS;
            b.cancel = dil::persist_cancel_word(c->pws);
            b.stop = dil::persist_stop_word(c->pws, k);
            e = dil::launch_sign_batch(x.level, dil::SIGN_PLAIN, b,
                                       static_cast<uint8_t *>(c->pws) + dil::PERSIST_HEADER_BYTES + k * p.region, st[k]);
        }
    }
    for (size_t k = 1; k < PIPE_STREAMS; ++k) {
        const cudaError_t r = cudaEventRecord(c->ev_join, st[k]), w = cudaStreamWaitEvent(s, c->ev_join, 0);
        if (e == cudaSuccess) e = r != cudaSuccess ? r : w;
    }
    return e;
}
}  // namespace

int dil_sign_persistent(dil_ctx *c, int njobs, const dil_sign_job *jobs, void *stream) {
    TraceRange trace("dil_sign_persistent");
    if (!c || njobs < 1 || njobs > dil::PERSIST_MAX_JOBS || !jobs) return DIL_EINVAL;
    dil::PersistJobs J;
    memset(&J, 0, sizeof(J));
    size_t total = 0;
    for (int j = 0; j < njobs; ++j) {
        const dil_sign_job &x = jobs[j];
        if (!level_ok(x.level)) return DIL_EINVAL;
        if (x.n && (!x.sk || !x.msg_off || !x.sig)) return DIL_EINVAL;
        J.job[j].level = x.level;
        J.job[j].n = (int)x.n;
        J.job[j].start = (int)total;
        J.job[j].sk = x.sk;
        J.job[j].msg = x.msg;
        J.job[j].off = x.msg_off;
        J.job[j].sig = x.sig;
        J.job[j].status = x.task_status;
        J.job[j].iters = x.iterations;
        total += x.n;
        if (total > (size_t)INT32_MAX / 2) return DIL_EINVAL;
    }
    J.njobs = njobs;
    J.total = (int)total;
    if (total == 0) return DIL_OK;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    // SMs per job in proportion to its work (a task's relative cost by level:
    // persistent Sign rates 3.65 / 2.42 / 1.98 M/s at 10,000 tasks)
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) return DIL_ECUDA;
    double w[dil::PERSIST_MAX_JOBS], sum = 0;
    for (int j = 0; j < njobs; ++j) {
        const int lv = J.job[j].level;
        w[j] = (double)J.job[j].n * (lv == 2 ? 1.0 : lv == 3 ? 1.51 : 1.84);
        sum += w[j];
    }
    double acc = 0;
    for (int j = 0; j < njobs; ++j) {
        acc += w[j];
        J.sm_end[j] = j + 1 == njobs ? (1 << 30) : (int)(sms * acc / sum + 0.5);
    }
    // One-warp launches run in rounds; shapes of two or four warps per task, device
    // memory too short for them, and the hook that makes bounded waits run out keep
    // the device queue.
    const bool wish = !(c->ptune_set && c->ptune.p > 1) && c->spin_limit == 0;
    const int max_iter = c->max_iter;
    if (!c->gexec || !same_jobs(J, c->gjobs) || !same_tune(c->ptune, c->gtune) || max_iter != c->gmax_iter ||
        c->spin_limit != c->gspin_limit || wish != c->gwish || c->gws != c->pws) {
        // (this also warms the attribute / occupancy queries outside the capture)
        const size_t queue = dil::persist_workspace_bytes(J, c->ptune, c->device);
        RoundPlan plan = wish ? planned_rounds(c, J, c->budget, queue) : RoundPlan{};
        if (plan.bytes == 0) {
            if (queue == 0) return DIL_ECUDA;
            const int rc = queue > c->budget ? DIL_ENOMEM : ensure_pws(c, queue);
            if (rc && wish) plan = planned_rounds(c, J, std::min(queue, c->budget), 0);
            if (rc && plan.bytes == 0) return rc;
        }
        const bool rounds = plan.bytes != 0;
        if (rounds) {
            const int rc = ensure_aux(c, PIPE_STREAMS - 1);
            if (rc) return rc;
        }
        if (c->gexec) {
            cudaGraphExecDestroy(c->gexec);
            c->gexec = nullptr;
        }
        if (!c->cap_stream && cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
            return DIL_ECUDA;
        cudaGraph_t graph = nullptr;
        if (cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) return DIL_ECUDA;
        cudaError_t e = rounds ? launch_rounds(c, J, plan, c->cap_stream)
                               : dil::launch_sign_persist(J, c->pws, c->ptune, max_iter, c->spin_limit, c->device,
                                                          c->cap_stream);
        cudaError_t e2 = cudaStreamEndCapture(c->cap_stream, &graph);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            cudaGetLastError();
            return DIL_ECUDA;
        }
        e = cudaGraphInstantiate(&c->gexec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            c->gexec = nullptr;
            return DIL_ECUDA;
        }
        c->gjobs = J;
        c->gtune = c->ptune;
        c->gmax_iter = max_iter;
        c->gspin_limit = c->spin_limit;
        c->gwish = wish;
        c->gws = c->pws;
    }
    return cudaGraphLaunch(c->gexec, (cudaStream_t)stream) == cudaSuccess ? DIL_OK : DIL_ECUDA;
}

int dil_persistent_status(dil_ctx *c, void *stream) {
    if (!c) return DIL_EINVAL;
    DeviceGuard g(c->device);
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return DIL_ECUDA;
    std::lock_guard<std::mutex> lk(c->mu);
    if (!c->pws) return DIL_OK;
    return dil::persist_error(c->pws);
}

int dil_persistent_cancel(dil_ctx *c) {
    TraceRange trace("dil_persistent_cancel");
    if (!c) return DIL_EINVAL;
    DeviceGuard g(c->device);
    std::lock_guard<std::mutex> lk(c->mu);
    if (!c->pws) return DIL_OK;
    if (!c->cancel_stream && cudaStreamCreateWithFlags(&c->cancel_stream, cudaStreamNonBlocking) != cudaSuccess)
        return DIL_ECUDA;
    return dil::persist_cancel(c->pws, c->cancel_stream) == cudaSuccess ? DIL_OK : DIL_ECUDA;
}

// ---------------------------------------------------------------- key stores
}  // extern "C"

extern "C" {

int dil_keystore_create(dil_ctx *c, int level, size_t n_keys, const uint8_t *pk, const uint8_t *sk,
                        dil_keystore **out, void *stream) {
    TraceRange trace("dil_keystore_create");
    if (!c || !out || !level_ok(level) || n_keys == 0 || !pk || n_keys > (size_t)INT32_MAX) return DIL_EINVAL;
    *out = nullptr;
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    DeviceGuard g(c->device);
    dil_keystore *ks = new dil_keystore;
    ks->device = c->device;
    ks->level = level;
    ks->n = n_keys;
    const size_t kbytes = n_keys * dil::key_polys(level) * POLY_BYTES;
    bool okm = cudaMalloc(&ks->pk, pkb * n_keys) == cudaSuccess && cudaMalloc(&ks->tr, 32 * n_keys) == cudaSuccess &&
               cudaMalloc(&ks->keys, kbytes) == cudaSuccess;
    if (okm && sk) okm = cudaMalloc(&ks->sk, skb * n_keys) == cudaSuccess;
    if (!okm) {
        cudaGetLastError();
        dil_keystore_destroy(ks);
        return DIL_ENOMEM;
    }
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(ks->pk, pk, pkb * n_keys, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess && sk) e = cudaMemcpyAsync(ks->sk, sk, skb * n_keys, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess)
        e = dil::launch_key_prepare(level, (int)n_keys, ks->pk, ks->sk, ks->keys, ks->tr, 8, 2, s);
    if (e != cudaSuccess) {
        dil_keystore_destroy(ks);
        return cuda_fail(e);
    }
    *out = ks;
    return DIL_OK;
}

int dil_keystore_destroy(dil_keystore *ks) {
    if (!ks) return DIL_OK;
    {
        DeviceGuard g(ks->device);
        cudaDeviceSynchronize();
        if (ks->pk) cudaFree(ks->pk);
        if (ks->sk) cudaFree(ks->sk);
        if (ks->tr) cudaFree(ks->tr);
        if (ks->keys) cudaFree(ks->keys);
    }
    delete ks;
    return DIL_OK;
}

int dil_sign_keyed(dil_ctx *c, const dil_keystore *ks, size_t n, const int32_t *key_idx, const uint8_t *msg,
                   const uint64_t *msg_off, uint8_t *sig, int32_t *task_status, void *stream) {
    TraceRange trace("dil_sign_keyed");
    if (!c || !ks || !ks->sk || ks->device != c->device) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!key_idx || !msg_off || !sig || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(ks->level, pkb, skb, sigb);
    const int max_iter = sign_cap(c, ks->level);
    if (!sign_fused(c, ks->level, dil::SIGN_KEYED)) {
        dil::SignBatch b{};
        b.sk = ks->sk;
        b.msg = msg;
        b.off = msg_off;
        b.sig = sig;
        b.status = task_status;
        b.keys = ks->keys;
        b.key_idx = key_idx;
        b.n_keys = (int)ks->n;
        b.max_iter = max_iter;
        return run_sign_batch(c, ks->level, dil::SIGN_KEYED, n, b, (cudaStream_t)stream);
    }
    const size_t per = dil::keyed_sign_polys(ks->level) * POLY_BYTES;
    size_t chunk = std::min<size_t>(n, c->budget / per);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * per);
    if (rc) return rc;
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        int m = (int)std::min(chunk, n - s0);
        cudaError_t e = dil::launch_sign_keyed(ks->level, m, (int)ks->n, key_idx + s0, ks->sk, ks->keys, msg,
                                               msg_off + s0, sig + sigb * s0,
                                               task_status ? task_status + s0 : nullptr, nullptr, (int32_t *)c->ws,
                                               max_iter, fused_warps(c, 1, ks->level), fused_wpt(c, 1, ks->level),
                                               (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    return DIL_OK;
}

int dil_verify_keyed(dil_ctx *c, const dil_keystore *ks, size_t n, const int32_t *key_idx, const uint8_t *msg,
                     const uint64_t *msg_off, const uint8_t *sig, uint8_t *ok, void *stream) {
    TraceRange trace("dil_verify_keyed");
    if (!c || !ks || ks->device != c->device) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!key_idx || !msg_off || !sig || !ok || n > (size_t)INT32_MAX) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    size_t pkb, skb, sigb;
    sizes_of(ks->level, pkb, skb, sigb);
    const Shape sh = shape_of(c, 2, ks->level);
    if (!sh.fused) {
        dil::VerifyBatch b{};
        b.pk = ks->pk;
        b.msg = msg;
        b.off = msg_off;
        b.sig = sig;
        b.ok = ok;
        b.keys = ks->keys;
        b.key_idx = key_idx;
        b.key_tr = ks->tr;
        b.n_keys = (int)ks->n;
        return run_verify_batch(c, ks->level, dil::VERIFY_KEYED, n, b, (cudaStream_t)stream);
    }
    const size_t per = dil::keyed_verify_polys(ks->level) * POLY_BYTES;
    size_t chunk = chunk_tasks(c, per, n);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * per);
    if (rc) return rc;
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        int m = (int)std::min(chunk, n - s0);
        cudaError_t e = dil::launch_verify_keyed(ks->level, m, (int)ks->n, key_idx + s0, ks->pk, ks->keys, ks->tr, msg,
                                                 msg_off + s0, sig + sigb * s0, ok + s0, (int32_t *)c->ws, sh.warps,
                                                 sh.p, (cudaStream_t)stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    return DIL_OK;
}

}  // extern "C"

// ---------------------------------------------------------------- host forms
namespace {

// Device staging for the host forms: grows on demand (not part of the budget).
int ensure_stage(dil_ctx *c, size_t bytes) {
    if (bytes <= c->stage_bytes) return DIL_OK;
    if (c->stage) {
        cudaDeviceSynchronize();
        cudaFree(c->stage);
        c->stage = nullptr;
        c->stage_bytes = 0;
    }
    if (cudaMalloc(&c->stage, bytes) != cudaSuccess) {
        cudaGetLastError();
        return DIL_ENOMEM;
    }
    c->stage_bytes = bytes;
    return DIL_OK;
}

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// Host-buffer forms as a pipeline (the paper's section 4.4 multi-stream
// overlap): a large batch is cut into PIPE_STREAMS chunks, each on its own
// stream (the caller's and the context's extra ones) with its own part of the
// workspace.  A chunk copies its inputs in, runs its kernel and copies its
// outputs back; the chunks' kernels run concurrently (together they fill the
// GPU like one launch, and their tails overlap), while the copies of one
// chunk overlap the kernels of the others.  When the budget cannot hold the
// whole batch's scratch, chunks shrink and cycle over the streams.

size_t pipe_streams(size_t n) { return n >= PIPE_MIN_TASKS ? PIPE_STREAMS : 1; }

// Tasks of a chunk whose kernel scratch is `per_task` bytes each (0: does not fit).
size_t pipe_tasks(const dil_ctx *c, size_t n, size_t per_task) {
    const size_t ns = pipe_streams(n);
    return std::min((n + ns - 1) / ns, c->budget / (ns * per_task));
}

// run_streams, and a wait for the caller's stream.
template <class Chunk>
int run_pipeline(dil_ctx *c, size_t n, size_t per, size_t region, cudaStream_t s0, Chunk chunk) {
    const int rc = run_streams(c, n, per, region, pipe_streams(n), s0, chunk);
    const cudaError_t e = cudaStreamSynchronize(s0);
    if (rc) return rc;
    return e == cudaSuccess ? DIL_OK : DIL_ECUDA;
}

// Host offsets of the host forms: non-decreasing (a task's message is
// msg[off[i] .. off[i + 1])).
bool offsets_ok(const uint64_t *off, size_t n) {
    for (size_t i = 0; i < n; ++i)
        if (off[i + 1] < off[i]) return false;
    return true;
}

bool h2d(void *dst, const void *src, size_t bytes, cudaStream_t s) {
    return bytes == 0 || cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s) == cudaSuccess;
}
bool d2h(void *dst, const void *src, size_t bytes, cudaStream_t s) {
    return bytes == 0 || cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s) == cudaSuccess;
}

}  // namespace

extern "C" {

int dil_keygen_host(dil_ctx *c, int level, size_t n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk,
                    void *stream) {
    TraceRange trace("dil_keygen_host");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!seeds || !pk || !sk || n > (size_t)INT32_MAX) return DIL_EINVAL;
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    int rc = ensure_stage(c, al(32 * n) + al(pkb * n) + al(skb * n));
    if (rc) return rc;
    uint8_t *d_seed = (uint8_t *)c->stage, *d_pk = d_seed + al(32 * n), *d_sk = d_pk + al(pkb * n);
    const size_t per = dil::scratch_polys(dil::OP_KEYGEN, level) * POLY_BYTES;
    const Shape sh = shape_of(c, 0, level);
    const size_t tasks = pipe_tasks(c, n, per);
    return run_pipeline(c, n, tasks, tasks * per, (cudaStream_t)stream,
                        [&](size_t c0, size_t c1, cudaStream_t s, int32_t *scratch) -> int {
                            const size_t m = c1 - c0;
                            if (!h2d(d_seed + 32 * c0, seeds + 32 * c0, 32 * m, s)) return DIL_ECUDA;
                            cudaError_t e = keygen_chunk(sh, level, (int)m, d_seed + 32 * c0, d_pk + pkb * c0,
                                                         d_sk + skb * c0, scratch, s);
                            if (e != cudaSuccess) return cuda_fail(e);
                            if (!d2h(pk + pkb * c0, d_pk + pkb * c0, pkb * m, s) ||
                                !d2h(sk + skb * c0, d_sk + skb * c0, skb * m, s))
                                return DIL_ECUDA;
                            return DIL_OK;
                        });
}

int dil_sign_host(dil_ctx *c, int level, size_t n, const uint8_t *sk, const uint8_t *msg, const uint64_t *msg_off,
                  uint8_t *sig, int32_t *task_status, void *stream) {
    TraceRange trace("dil_sign_host");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!sk || !msg_off || !sig || n > (size_t)INT32_MAX) return DIL_EINVAL;
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const size_t mlen = (size_t)msg_off[n];
    if ((mlen && !msg) || !offsets_ok(msg_off, n)) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    int rc = ensure_stage(c, al(skb * n) + al(mlen + 1) + al(8 * (n + 1)) + al(sigb * n) + al(4 * n));
    if (rc) return rc;
    uint8_t *d_sk = (uint8_t *)c->stage, *d_msg = d_sk + al(skb * n);
    uint64_t *d_off = (uint64_t *)(d_msg + al(mlen + 1));
    uint8_t *d_sig = (uint8_t *)d_off + al(8 * (n + 1));
    int32_t *d_st = (int32_t *)(d_sig + al(sigb * n));
    const int max_iter = sign_cap(c, level);
    const size_t ns = pipe_streams(n);
    const RoundSize z = c->wpt[1][lidx(level)] > 1 ? RoundSize{0, 0}
                                                   : round_size(level, dil::SIGN_PLAIN, (n + ns - 1) / ns,
                                                                c->budget / ns, (int)ns);
    const size_t fused = dil::scratch_polys(dil::OP_SIGN, level) * POLY_BYTES;
    const size_t tasks = z.tasks ? z.tasks : pipe_tasks(c, n, fused);
    const size_t region = z.tasks ? dil::sign_batch_bytes(level, dil::SIGN_PLAIN, z.tasks, z.slots) : tasks * fused;
    return run_pipeline(c, n, tasks, region, (cudaStream_t)stream,
                        [&](size_t c0, size_t c1, cudaStream_t s, int32_t *scratch) -> int {
                            const size_t m = c1 - c0;
                            if (!h2d(d_sk + skb * c0, sk + skb * c0, skb * m, s) ||
                                !h2d(d_msg + msg_off[c0], msg ? msg + msg_off[c0] : nullptr,
                                     (size_t)(msg_off[c1] - msg_off[c0]), s) ||
                                !h2d(d_off + c0, msg_off + c0, 8 * (m + 1), s))
                                return DIL_ECUDA;
                            cudaError_t e;
                            if (z.tasks) {
                                dil::SignBatch b{};
                                b.n = (int)m;
                                b.slots = (int)z.slots;
                                b.parts = (int)ns;
                                b.on_gpu = (int)std::min(n, ns * z.tasks);
                                b.sk = d_sk + skb * c0;
                                b.msg = d_msg;
                                b.off = d_off + c0;
                                b.sig = d_sig + sigb * c0;
                                b.status = d_st + c0;
                                b.max_iter = max_iter;
                                e = dil::launch_sign_batch(level, dil::SIGN_PLAIN, b, scratch, s);
                            } else {
                                e = dil::launch_sign(level, (int)m, d_sk + skb * c0, d_msg, d_off + c0,
                                                     d_sig + sigb * c0, d_st + c0, nullptr, scratch, max_iter,
                                                     fused_warps(c, 1, level), fused_wpt(c, 1, level), s);
                            }
                            if (e != cudaSuccess) return cuda_fail(e);
                            if (!d2h(sig + sigb * c0, d_sig + sigb * c0, sigb * m, s) ||
                                (task_status && !d2h(task_status + c0, d_st + c0, 4 * m, s)))
                                return DIL_ECUDA;
                            return DIL_OK;
                        });
}

int dil_verify_host(dil_ctx *c, int level, size_t n, const uint8_t *pk, const uint8_t *msg,
                    const uint64_t *msg_off, const uint8_t *sig, uint8_t *ok, void *stream) {
    TraceRange trace("dil_verify_host");
    if (!c || !level_ok(level)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!pk || !msg_off || !sig || !ok || n > (size_t)INT32_MAX) return DIL_EINVAL;
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const size_t mlen = (size_t)msg_off[n];
    if ((mlen && !msg) || !offsets_ok(msg_off, n)) return DIL_EINVAL;
    std::lock_guard<std::mutex> lk(c->mu);
    DeviceGuard g(c->device);
    int rc = ensure_stage(c, al(pkb * n) + al(mlen + 1) + al(8 * (n + 1)) + al(sigb * n) + al(n));
    if (rc) return rc;
    uint8_t *d_pk = (uint8_t *)c->stage, *d_msg = d_pk + al(pkb * n);
    uint64_t *d_off = (uint64_t *)(d_msg + al(mlen + 1));
    uint8_t *d_sig = (uint8_t *)d_off + al(8 * (n + 1));
    uint8_t *d_ok = d_sig + al(sigb * n);
    const size_t batch = verify_task_bytes(level, dil::VERIFY_PLAIN);
    const Shape sh = shape_of(c, 2, level);
    const size_t per = sh.fused ? dil::scratch_polys(dil::OP_VERIFY, level) * POLY_BYTES : batch;
    const size_t tasks = pipe_tasks(c, n, per);
    // one chunk at a time: its hashes run beside the rest, as in dil_verify (1,000
    // Dilithium3 tasks 250 -> 196 us); of four chunks, each beside the others
    dil::VerifyFork fork{};
    if (!sh.fused && pipe_streams(n) == 1) {
        if ((rc = ensure_aux(c, 1))) return rc;
        fork = {c->aux[0], c->ev_fork, c->ev_join};
    }
    return run_pipeline(c, n, tasks, tasks * per, (cudaStream_t)stream,
                        [&](size_t c0, size_t c1, cudaStream_t s, int32_t *scratch) -> int {
                            const size_t m = c1 - c0;
                            if (!h2d(d_pk + pkb * c0, pk + pkb * c0, pkb * m, s) ||
                                !h2d(d_msg + msg_off[c0], msg ? msg + msg_off[c0] : nullptr,
                                     (size_t)(msg_off[c1] - msg_off[c0]), s) ||
                                !h2d(d_off + c0, msg_off + c0, 8 * (m + 1), s) ||
                                !h2d(d_sig + sigb * c0, sig + sigb * c0, sigb * m, s))
                                return DIL_ECUDA;
                            cudaError_t e;
                            if (sh.fused) {
                                e = dil::launch_verify(level, (int)m, d_pk + pkb * c0, d_msg, d_off + c0,
                                                       d_sig + sigb * c0, d_ok + c0, scratch, sh.warps, sh.p, s);
                            } else {
                                dil::VerifyBatch b{};
                                carve_verify(b, scratch, m, dil::verify_batch_polys(level, dil::VERIFY_PLAIN));
                                b.pk = d_pk + pkb * c0;
                                b.msg = d_msg;
                                b.off = d_off + c0;
                                b.sig = d_sig + sigb * c0;
                                b.ok = d_ok + c0;
                                e = dil::launch_verify_batch(level, dil::VERIFY_PLAIN, b, fork, s);
                            }
                            if (e != cudaSuccess) return cuda_fail(e);
                            if (!d2h(ok + c0, d_ok + c0, m, s)) return DIL_ECUDA;
                            return DIL_OK;
                        });
}

// ---------------------------------------------------------------- test-only
#define TEST_PROLOGUE(ctx)                  \
    if (!(ctx)) return DIL_EINVAL;          \
    std::lock_guard<std::mutex> lk((ctx)->mu); \
    DeviceGuard g((ctx)->device);

static int status_of(cudaError_t e) { return e == cudaSuccess ? DIL_OK : cuda_fail(e); }

int dil_test_shake(dil_ctx *c, int kind, size_t n, const uint8_t *in, const uint64_t *in_off, uint8_t *out,
                   size_t outlen, void *stream) {
    TEST_PROLOGUE(c)
    if ((kind != 128 && kind != 256) || n > (size_t)INT32_MAX || outlen > (1u << 20)) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!in_off || !out) return DIL_EINVAL;
    return status_of(dil::launch_test_shake(kind, (int)n, in, in_off, out, (int)outlen, (cudaStream_t)stream));
}

int dil_test_k16_rider(dil_ctx *c, size_t n, const uint8_t *in, const uint64_t *in_off, const int32_t *perms,
                       uint8_t *out, void *stream) {
    TEST_PROLOGUE(c)
    if (n > (size_t)INT32_MAX) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!in_off || !perms || !out) return DIL_EINVAL;
    return status_of(dil::launch_test_k16_rider((int)n, in, in_off, perms, out, (cudaStream_t)stream));
}

int dil_test_k16_chain_rider(dil_ctx *c, size_t n, const uint8_t *in, const uint64_t *in_off, const int32_t *perms,
                             const int32_t *step, uint8_t *out, void *stream) {
    TEST_PROLOGUE(c)
    if (n > (size_t)INT32_MAX) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!in_off || !perms || !step || !out) return DIL_EINVAL;
    return status_of(dil::launch_test_k16_chain_rider((int)n, in, in_off, perms, step, out, (cudaStream_t)stream));
}

int dil_test_keccak_f(dil_ctx *c, int form, size_t n, const uint64_t *in, uint64_t *out, void *stream) {
    TEST_PROLOGUE(c)
    if ((form != 1 && form != 2 && form != 6 && form != 16) || n > (size_t)INT32_MAX) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!in || !out) return DIL_EINVAL;
    return status_of(dil::launch_test_keccak_f(form, (int)n, in, out, (cudaStream_t)stream));
}

int dil_test_t0_ntt(dil_ctx *c, int level, int variant, size_t n, const uint8_t *sk, int32_t *t0hat, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || variant < 0 || variant > 3 || n > (size_t)INT32_MAX) return DIL_EINVAL;
    if (n == 0) return DIL_OK;
    if (!sk || !t0hat) return DIL_EINVAL;
    int32_t *tmp = nullptr;
    if (variant <= 1) {
        const size_t k = level == 2 ? 4 : level == 3 ? 6 : 8;
        const int rc = ensure_ws(c, n * k * POLY_BYTES);
        if (rc) return rc;
        tmp = static_cast<int32_t *>(c->ws);
    }
    return status_of(dil::launch_test_t0_ntt(level, variant, (int)n, sk, tmp, t0hat, (cudaStream_t)stream));
}

int dil_test_ntt(dil_ctx *c, size_t n, const int32_t *in, int32_t *out, int inverse, void *stream) {
    TEST_PROLOGUE(c)
    if (n > (size_t)INT32_MAX || (n && (!in || !out))) return DIL_EINVAL;
    return status_of(dil::launch_test_ntt((int)n, in, out, inverse ? 1 : 0, (cudaStream_t)stream));
}

int dil_test_expand_a(dil_ctx *c, int level, size_t n, const uint8_t *rho, int32_t *ahat, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!rho || !ahat))) return DIL_EINVAL;
    return status_of(dil::launch_test_expand_a(level, (int)n, rho, ahat, (cudaStream_t)stream));
}

int dil_test_expand_a_refill(dil_ctx *c, int level, size_t n, const uint8_t *rho, int lane_order, int32_t *ahat,
                             void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!rho || !ahat))) return DIL_EINVAL;
    return status_of(dil::launch_test_expand_a_refill(level, (int)n, rho, !lane_order, ahat, (cudaStream_t)stream));
}

int dil_test_expand_s(dil_ctx *c, int level, size_t n, const uint8_t *rhop, int32_t *s, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!rhop || !s))) return DIL_EINVAL;
    return status_of(dil::launch_test_expand_s(level, (int)n, rhop, s, (cudaStream_t)stream));
}

int dil_test_expand_mask(dil_ctx *c, int level, size_t n, const uint8_t *rhop, const int32_t *kappa, int32_t *y,
                         void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!rhop || !kappa || !y))) return DIL_EINVAL;
    return status_of(dil::launch_test_expand_mask(level, (int)n, rhop, kappa, y, (cudaStream_t)stream));
}

int dil_test_sample_in_ball_stream(dil_ctx *c, int level, size_t n, const uint8_t *bytes, int blocks, int32_t *cc,
                                   void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || blocks < 1 || blocks > 64 || (n && (!bytes || !cc)))
        return DIL_EINVAL;
    return status_of(dil::launch_test_sib_stream(level, (int)n, bytes, blocks, cc, (cudaStream_t)stream));
}

int dil_test_sample_in_ball(dil_ctx *c, int level, size_t n, const uint8_t *ctilde, int32_t *cc, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!ctilde || !cc))) return DIL_EINVAL;
    return status_of(dil::launch_test_sample_in_ball(level, (int)n, ctilde, cc, (cudaStream_t)stream));
}

int dil_test_rounding(dil_ctx *c, int level, size_t n, const int32_t *r, const int32_t *z, const uint8_t *h,
                      int32_t *out, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level) || n > (size_t)INT32_MAX || (n && (!r || !z || !h || !out))) return DIL_EINVAL;
    return status_of(dil::launch_test_rounding(level, (int)n, r, z, h, out, (cudaStream_t)stream));
}

int dil_test_bounded_wait(dil_ctx *c, int flag_value, int limit, int *result) {
    TEST_PROLOGUE(c)
    if (!result || limit < 1 || limit > (1 << 24)) return DIL_EINVAL;
    return status_of(dil::test_bounded_wait(flag_value, limit, result));
}

int dil_test_set_spin_limit(dil_ctx *c, int limit) {
    TEST_PROLOGUE(c)
    if (limit < 0 || limit > dil::PERSIST_SPIN_LIMIT) return DIL_EINVAL;
    c->spin_limit = limit;
    return DIL_OK;
}

int dil_test_set_alloc_limit(dil_ctx *c, size_t bytes) {
    TEST_PROLOGUE(c)
    c->alloc_limit = bytes;
    return DIL_OK;
}

int dil_test_issue_rate(dil_ctx *c, int op, double *thread_ops_per_sm_clk) {
    TEST_PROLOGUE(c)
    if (op < 0 || op > 4 || !thread_ops_per_sm_clk) return DIL_EINVAL;
    return status_of(dil::measure_issue_rate(op, thread_ops_per_sm_clk));
}

int dil_test_sign_split(dil_ctx *c, int level, size_t n, const uint8_t *sk, const uint8_t *msg,
                        const uint64_t *msg_off, uint8_t *sig, int32_t *task_status, int32_t *iterations,
                        int *rounds, void *stream) {
    TEST_PROLOGUE(c)
    if (!level_ok(level)) return DIL_EINVAL;
    if (rounds) *rounds = 0;
    if (n == 0) return DIL_OK;
    if (!sk || !msg_off || !sig || n > (size_t)INT32_MAX) return DIL_EINVAL;
    size_t pkb, skb, sigb;
    sizes_of(level, pkb, skb, sigb);
    const int l = level == 2 ? 4 : level == 3 ? 5 : 7, cap = (65536 - l) / l + 1;
    const int max_iter = (c->max_iter > 0 && c->max_iter < cap) ? c->max_iter : cap;
    const int p = std::min(fused_wpt(c, 1, level), 2), w = std::max(fused_warps(c, 1, level) / p * p, p);
    const size_t per = dil::scratch_polys(dil::OP_SIGN, level) * POLY_BYTES + dil::split_state_bytes();
    const size_t chunk = std::min<size_t>(n, (c->budget - 256) / per);
    if (chunk == 0) return DIL_ENOMEM;
    int rc = ensure_ws(c, chunk * per + 256);
    if (rc) return rc;
    int32_t *scratch = (int32_t *)c->ws;
    void *state = (uint8_t *)c->ws + chunk * dil::scratch_polys(dil::OP_SIGN, level) * POLY_BYTES;
    int *pending = (int *)((uint8_t *)state + chunk * dil::split_state_bytes());
    for (size_t s0 = 0; s0 < n; s0 += chunk) {
        const int m = (int)std::min(chunk, n - s0);
        int r = 0;
        cudaError_t e = dil::launch_sign_split(level, m, sk + skb * s0, msg, msg_off + s0, sig + sigb * s0,
                                               task_status ? task_status + s0 : nullptr,
                                               iterations ? iterations + s0 : nullptr, scratch, state, pending,
                                               max_iter, w, p, (cudaStream_t)stream, &r);
        if (e != cudaSuccess) return cuda_fail(e);
        if (rounds) *rounds = std::max(*rounds, r);
    }
    return DIL_OK;
}

int dil_test_keccak_rate(dil_ctx *c, int form, double *sm_clocks_per_state_round) {
    TEST_PROLOGUE(c)
    if ((form != 1 && form != 2 && form != 6 && form != 16) || !sm_clocks_per_state_round) return DIL_EINVAL;
    return status_of(dil::measure_keccak_rate(form, sm_clocks_per_state_round));
}

}  // extern "C"
