// Batched PNE / HPNE (Alg. 1 on many independent problems of uneven shape).
//
// The problems are spread over a fixed set of internal streams (heaviest
// first, each to the least-loaded stream).  A batch seen for the first time is
// enqueued there, forked from and joined to the caller's stream by events; when the
// same batch (descriptors, workspace, settings) comes again the whole fan-out -- every
// kernel of every problem plus the fork/join events -- is captured into one CUDA
// graph, and from then on a call is one graph launch on the caller's stream.
// Problems asking for the AUTO
// precision first get one batched condition-estimate pass (Sec. 6.1; on A^T A
// for AUTO, on a sketch for AUTO_SKETCH) and a single readback of the chosen
// precisions, because kernel selection in the captured graph needs them on
// the host.  The batched sketch and preconditioner QR (lsq_sketch_batched,
// lsq_precond_qr_batched) use the same fan-out.
#include "common.cuh"
#include "kernels.cuh"

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <optional>
#include <vector>

namespace lsq {
lsq_status solve_impl_ext(bool hpne, const double* A, int64_t m, int64_t n, int64_t lda, const double* b,
                          const lsq_opts* o, double* x, double* Rs_out, int32_t* info, void* ws, size_t ws_bytes,
                          cudaStream_t st, const double* Rs_in);
size_t solve_ws_bytes_ext(int64_t m, int64_t n, const lsq_opts* o, bool hpne);
lsq_status check_opts_ext(const lsq_opts* o, int64_t m, int64_t n);
}  // namespace lsq

namespace {

using namespace lsq;

constexpr int kMaxStreams = 64;

// Internal streams of the fan-out: 16, or $LSQ_BATCH_STREAMS (1 .. 64), read
// once per process.
int n_streams() {
    static const int ns = [] {
        const char* e = std::getenv("LSQ_BATCH_STREAMS");
        const int v = e ? std::atoi(e) : 16;
        return v < 1 ? 1 : (v > kMaxStreams ? kMaxStreams : v);
    }();
    return ns;
}

struct BatchState {
    std::mutex mu;
    int dev = -1;
    cudaStream_t sub[kMaxStreams] = {};
    cudaStream_t cap = nullptr;  // the graph is captured here, never on the caller stream
    cudaEvent_t fork = nullptr;
    cudaEvent_t join[kMaxStreams] = {};
};
BatchState g_batch;

// A cached executable graph and the description it was built from: one for
// the solves (or the batched sketch / QR steps), one for the estimate pass.
struct GraphCache {
    cudaGraphExec_t exec = nullptr;
    std::vector<unsigned char> key;
    std::vector<unsigned char> seen;  // of the last batch that was enqueued without a graph
    void drop() {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        key.clear();
    }
};
GraphCache g_main, g_est;
lsq_status ensure_streams() {
    int dev = 0;
    LSQ_CUDA_TRY(cudaGetDevice(&dev));
    if (g_batch.dev == dev && g_batch.fork) return LSQ_OK;
    for (int k = 0; k < n_streams(); ++k) {
        LSQ_CUDA_TRY(cudaStreamCreateWithFlags(&g_batch.sub[k], cudaStreamNonBlocking));
        LSQ_CUDA_TRY(cudaEventCreateWithFlags(&g_batch.join[k], cudaEventDisableTiming));
    }
    LSQ_CUDA_TRY(cudaEventCreateWithFlags(&g_batch.fork, cudaEventDisableTiming));
    LSQ_CUDA_TRY(cudaStreamCreateWithFlags(&g_batch.cap, cudaStreamNonBlocking));
    g_batch.dev = dev;
    for (GraphCache* c : {&g_main, &g_est}) {
        c->drop();
        c->seen.clear();
    }
    return LSQ_OK;
}

// What the kernels of a fan-out depend on beside its descriptors, at the end of
// its graph's key: the buffers, which call it is (tag) and the library's switches
// and reduction hook (a captured hook is part of the graph).
void key_tail(std::vector<unsigned char>& key, const void* ws, size_t ws_bytes, int tag) {
    struct Tail {
        const void* ws;
        uint64_t ws_bytes;
        int64_t tag, emulation, tc_sketch;
        uint64_t wait_ns;
        const void *hook, *hook_user;
    } t{ws, ws_bytes, tag, fp64_emulation_enabled() ? 1 : 0, tensor_core_sketch_enabled() ? 1 : 0, trsv_wait_ns(), nullptr,
        nullptr};
    reduce_hook(&t.hook, &t.hook_user);
    static_assert(sizeof(Tail) == 64, "no padding");
    key.insert(key.end(), (const unsigned char*)&t, (const unsigned char*)&t + sizeof(t));
}

struct Plan {
    std::vector<int> stream_of;   // problem -> internal stream
    std::vector<int> order;       // launch order (heaviest first)
    size_t slot_bytes = 0;        // workspace per internal stream
    size_t head_bytes = 0;        // chosen-precision scratch at the front
};

double work_of(const lsq_batch_problem& p) { return 2.0 * (double)p.m * (double)p.n * (double)p.n; }

Plan make_plan(bool hpne, int32_t count, const lsq_batch_problem* probs) {
    Plan P;
    P.stream_of.assign(count, 0);
    P.order.resize(count);
    for (int i = 0; i < count; ++i) P.order[i] = i;
    std::stable_sort(P.order.begin(), P.order.end(),
                     [&](int a, int b) { return work_of(probs[a]) > work_of(probs[b]); });
    double load[kMaxStreams] = {};
    for (int i : P.order) {
        int best = 0;
        for (int k = 1; k < n_streams(); ++k)
            if (load[k] < load[best]) best = k;
        P.stream_of[i] = best;
        load[best] += work_of(probs[i]);
    }
    for (int i = 0; i < count; ++i) {
        size_t need = solve_ws_bytes_ext(probs[i].m, probs[i].n, &probs[i].opts, hpne);
        size_t c = condest_ws_bytes(probs[i].m, probs[i].n, device_sm_count());
        if (probs[i].opts.sketch_prec == LSQ_AUTO_SKETCH)
            c = std::max(c, lsq_workspace_size(LSQ_OP_CONDEST_SKETCH, probs[i].m, probs[i].n, nullptr));
        P.slot_bytes = std::max(P.slot_bytes, std::max(need, c));
    }
    P.slot_bytes = align_up(P.slot_bytes, 256);
    P.head_bytes = align_up((size_t)count * (sizeof(double) + sizeof(int32_t)) + 512, 256);
    return P;
}

lsq_status check_problem(const lsq_batch_problem& p) {
    if (!p.A || !p.b || !p.x || !p.info || p.m <= 0 || p.n <= 0 || p.lda < p.m) return LSQ_ERR_ARG;
    const lsq_opts* o = &p.opts;
    if (o->kind != LSQ_GAUSSIAN && o->kind != LSQ_SPARSE_SIGN && o->kind != LSQ_SRFT) return LSQ_ERR_ARG;
    if (o->s < p.n || o->s > p.m) return LSQ_ERR_ARG;
    if (o->kind == LSQ_SPARSE_SIGN && (o->zeta < 1 || o->zeta > 32 || o->zeta > o->s)) return LSQ_ERR_ARG;
    if (o->sketch_prec < LSQ_FP8_E4M3 || o->sketch_prec > LSQ_AUTO_SKETCH) return LSQ_ERR_ARG;
    return LSQ_OK;
}

bool is_auto(int p) { return p == LSQ_AUTO || p == LSQ_AUTO_SKETCH; }

// The fan-out on the internal streams, forked from and joined to `from` by
// events: captured into a graph when `from` is being captured, else enqueued.
template <typename F>
lsq_status enqueue_fanout(cudaStream_t from, const std::vector<int>& order, const std::vector<int>& stream_of,
                          char* slots, size_t slot_bytes, F run) {
    lsq_status r = LSQ_OK;
    if (cudaEventRecord(g_batch.fork, from) != cudaSuccess) return LSQ_ERR_CUDA;
    for (int k = 0; k < n_streams() && r == LSQ_OK; ++k)
        if (cudaStreamWaitEvent(g_batch.sub[k], g_batch.fork, 0) != cudaSuccess) r = LSQ_ERR_CUDA;
    for (int i : order) {
        if (r != LSQ_OK) break;
        int k = stream_of[i];
        r = run(i, g_batch.sub[k], slots + (size_t)k * slot_bytes);
    }
    // joined after a failure too: what was enqueued uses the caller's buffers
    for (int k = 0; k < n_streams(); ++k)
        if ((cudaEventRecord(g_batch.join[k], g_batch.sub[k]) != cudaSuccess ||
             cudaStreamWaitEvent(from, g_batch.join[k], 0) != cudaSuccess) &&
            r == LSQ_OK)
            r = LSQ_ERR_CUDA;
    return r;
}

// Whether a fan-out may be enqueued without a graph: not when the caller's own
// stream is being captured, nor while a reduction hook or the stage timing would
// see every step twice when it is captured behind.
bool direct_ok(cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return cap == cudaStreamCaptureStatusNone && !reduce_hook_set() && !profiling_on();
}

// A fan-out of per-problem work over the internal streams, run(i, stream, slot)
// enqueuing problem i, cached as a graph in `cache` under `key`.  A batch that is not
// the last call's is enqueued on the internal streams directly; when it comes again it
// is captured (large problems, mean work 2 m n^2 from 1e9, directly once more and
// captured while the GPU runs them); from then on the graph is launched on st.
// Capturing and instantiating the thousands of launches of 64 solves takes ~46 ms of
// host time, which the GPU waited for when every new batch was captured first, and which
// came on top of enqueuing it when it was captured behind.  64 problems, another batch
// each call, precision from the estimate on a sketch, captured first / behind / not:
// 2000 x 32 33 / 43 / 16 ms, 16000 x 250 106 / 75 / 52 ms, the uneven ones 145 / 111 / 93
// (94 when the same batch is repeated).
// No step of a problem forks onto the library's shared look-ahead streams here
// (FanoutScope; captured or not), so concurrent problems never share a stream and both
// ways run the same kernels.  Caller holds g_batch.mu.
template <typename F>
lsq_status capture_fanout(GraphCache& cache, const std::vector<int>& order, const std::vector<int>& stream_of,
                          char* slots, size_t slot_bytes, std::vector<unsigned char>& key, double mean_work,
                          cudaStream_t st, F run) {
    if (cache.exec && key == cache.key) {
        LSQ_CUDA_TRY(cudaGraphLaunch(cache.exec, st));
        return LSQ_OK;
    }
    FanoutScope scope;
    const bool first = key != cache.seen;
    const bool direct = direct_ok(st) && (first || mean_work >= 1e9);
    if (direct) {
        lsq_status r = enqueue_fanout(st, order, stream_of, slots, slot_bytes, run);
        if (r != LSQ_OK) return r;
        if (first) {
            cache.seen.swap(key);
            return LSQ_OK;
        }
    }
    cache.drop();
    cudaGraph_t graph = nullptr;
    // Capture on an internal stream (the caller may use the legacy default
    // stream, which cannot be captured); the graph is then launched on st.
    cudaStream_t cs = g_batch.cap;
    const cudaError_t eb = cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed);
    if (eb != cudaSuccess) {
        cudaGetLastError();
        note_cuda_error(eb);
        return direct ? LSQ_OK : LSQ_ERR_CUDA;  // enqueued: as below
    }
    std::optional<UncountedScope> uncounted;
    if (direct) uncounted.emplace();
    const lsq_status cap = enqueue_fanout(cs, order, stream_of, slots, slot_bytes, run);
    uncounted.reset();
    cudaError_t ec = cudaStreamEndCapture(cs, &graph);
    if (cap != LSQ_OK || ec != cudaSuccess || !graph) {
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();  // do not leave a capture error behind for the caller
        if (direct) return LSQ_OK;  // the work is enqueued; the next call tries to capture it again
        return cap != LSQ_OK ? cap : LSQ_ERR_CUDA;
    }
    cudaGraphExec_t exec = nullptr;
    cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ei != cudaSuccess) {
        cudaGetLastError();
        return direct ? LSQ_OK : LSQ_ERR_CUDA;
    }
    cache.exec = exec;
    cache.key.swap(key);
    if (!direct) LSQ_CUDA_TRY(cudaGraphLaunch(cache.exec, st));
    return LSQ_OK;
}

// Heaviest first, each to the least-loaded internal stream.
void assign_streams(const std::vector<double>& work, std::vector<int>& order, std::vector<int>& stream_of) {
    const int count = (int)work.size();
    order.resize(count);
    stream_of.assign(count, 0);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return work[a] > work[b]; });
    double load[kMaxStreams] = {};
    for (int i : order) {
        int best = 0;
        for (int k = 1; k < n_streams(); ++k)
            if (load[k] < load[best]) best = k;
        stream_of[i] = best;
        load[best] += work[i];
    }
}

lsq_status batched(bool hpne, int32_t count, const lsq_batch_problem* probs, void* ws, size_t ws_bytes,
                   cudaStream_t st) {
    if (count <= 0 || !probs) return LSQ_ERR_ARG;
    // everything that a single solve refuses, before any problem runs
    for (int i = 0; i < count; ++i) {
        lsq_status r = check_problem(probs[i]);
        if (r == LSQ_OK) r = check_opts_ext(&probs[i].opts, probs[i].m, probs[i].n);
        if (r != LSQ_OK) return r;
    }
    std::lock_guard<std::mutex> lk(g_batch.mu);
    lsq_status r = ensure_streams();
    if (r != LSQ_OK) return r;
    Plan P = make_plan(hpne, count, probs);
    char* base = (char*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    size_t need = P.head_bytes + P.slot_bytes * n_streams() + 256;
    if (!ws || need > ws_bytes) return LSQ_ERR_NOMEM;
    char* slots = base + P.head_bytes;
    int sms = device_sm_count();

    // resolve AUTO precisions: one batched estimate pass (a cached graph of
    // its own), one readback
    std::vector<lsq_batch_problem> q(probs, probs + count);
    bool any_auto = false;
    for (int i = 0; i < count; ++i) any_auto |= is_auto(q[i].opts.sketch_prec);
    if (any_auto) {
        double* k0 = (double*)base;
        int32_t* ch = (int32_t*)(base + align_up(sizeof(double) * count, 256));
        std::vector<int> est_order;
        for (int i : P.order)
            if (is_auto(q[i].opts.sketch_prec)) est_order.push_back(i);
        std::vector<unsigned char> ekey(sizeof(lsq_batch_problem) * count);
        std::memcpy(ekey.data(), probs, sizeof(lsq_batch_problem) * count);
        key_tail(ekey, ws, ws_bytes, 0);
        double ework = 0.0;
        for (int i : est_order) ework += work_of(q[i]);
        r = capture_fanout(g_est, est_order, P.stream_of, slots, P.slot_bytes, ekey, ework / (double)est_order.size(), st,
                           [&](int i, cudaStream_t sk, char* slot) {
                               if (q[i].opts.sketch_prec == LSQ_AUTO)
                                   return launch_condest(q[i].A, q[i].m, q[i].n, q[i].lda, k0 + i, ch + i, slot,
                                                         P.slot_bytes, sms, sk);
                               return lsq_condest_sketch(q[i].A, q[i].m, q[i].n, q[i].lda, q[i].opts.seed, k0 + i,
                                                         ch + i, slot, P.slot_bytes, sk);
                           });
        if (r != LSQ_OK) return r;
        std::vector<int32_t> host_ch(count, LSQ_FP64);
        LSQ_CUDA_TRY(cudaMemcpyAsync(host_ch.data(), ch, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, st));
        LSQ_CUDA_TRY(cudaStreamSynchronize(st));
        for (int i = 0; i < count; ++i)
            if (is_auto(q[i].opts.sketch_prec)) {
                int p = host_ch[i];
                q[i].opts.sketch_prec = (p >= LSQ_FP8_E4M3 && p <= LSQ_FP64) ? p : LSQ_FP64;
                if (q[i].opts.sketch_prec == LSQ_FP64) q[i].opts.qr_prec = LSQ_FP64;
                if ((r = check_opts_ext(&q[i].opts, q[i].m, q[i].n)) != LSQ_OK) return r;
            }
    }

    // key of the captured graph: the resolved descriptors, the buffers and the settings
    std::vector<unsigned char> key(sizeof(lsq_batch_problem) * count);
    std::memcpy(key.data(), q.data(), sizeof(lsq_batch_problem) * count);
    key_tail(key, ws, ws_bytes, hpne ? 1 : 0);
    double work = 0.0;
    for (int i = 0; i < count; ++i) work += work_of(q[i]);
    return capture_fanout(g_main, P.order, P.stream_of, slots, P.slot_bytes, key, work / count, st,
                          [&](int i, cudaStream_t sk, char* slot) {
                              return solve_impl_ext(hpne, q[i].A, q[i].m, q[i].n, q[i].lda, q[i].b, &q[i].opts,
                                                    q[i].x, nullptr, q[i].info, slot, P.slot_bytes, sk, nullptr);
                          });
}

// ---- batched sketch and preconditioner QR --------------------------------
size_t sketch_slot_bytes(const lsq_sketch_problem& p) { return lsq_workspace_size(LSQ_OP_SKETCH, p.m, p.n, &p.opts); }
size_t qr_slot_bytes(const lsq_qr_problem& p) { return lsq_workspace_size(LSQ_OP_PRECOND_QR, p.s, p.n, nullptr); }

lsq_status check_sketch_problem(const lsq_sketch_problem& p) {
    if (!p.A || !p.As || !p.colexp || p.m <= 0 || p.n <= 0 || p.lda < p.m || p.ldas < p.opts.s) return LSQ_ERR_ARG;
    if (p.opts.sketch_prec < LSQ_FP8_E4M3 || p.opts.sketch_prec > LSQ_FP64) return LSQ_ERR_ARG;
    return sketch_slot_bytes(p) ? check_opts_ext(&p.opts, p.m, p.n) : LSQ_ERR_ARG;
}

lsq_status check_qr_problem(const lsq_qr_problem& p) {
    if (!p.As || !p.Rs || !p.info || p.n <= 0 || p.s < p.n || p.ldas < p.s || p.ldr < p.n) return LSQ_ERR_ARG;
    if ((p.as_prec != LSQ_FP32 && p.as_prec != LSQ_FP64) || (p.qr_prec != LSQ_FP32 && p.qr_prec != LSQ_FP64))
        return LSQ_ERR_ARG;
    return LSQ_OK;
}

template <typename Prob, typename Check, typename Slot, typename Work, typename Run>
lsq_status batched_steps(int tag, int32_t count, const Prob* probs, void* ws, size_t ws_bytes, cudaStream_t st,
                         Check check, Slot slot_of, Work work_of_p, Run run) {
    if (count <= 0 || !probs) return LSQ_ERR_ARG;
    size_t slot = 0;
    std::vector<double> work(count);
    for (int i = 0; i < count; ++i) {
        lsq_status r = check(probs[i]);
        if (r != LSQ_OK) return r;
        slot = std::max(slot, slot_of(probs[i]));
        work[i] = work_of_p(probs[i]);
    }
    slot = align_up(slot, 256);
    char* base = (char*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    if (!ws || slot * n_streams() + 512 > ws_bytes) return LSQ_ERR_NOMEM;
    std::lock_guard<std::mutex> lk(g_batch.mu);
    lsq_status r = ensure_streams();
    if (r != LSQ_OK) return r;
    std::vector<int> order, stream_of;
    assign_streams(work, order, stream_of);
    std::vector<unsigned char> key(sizeof(Prob) * count);
    std::memcpy(key.data(), probs, sizeof(Prob) * count);
    key_tail(key, ws, ws_bytes, tag);
    double sum = 0.0;
    for (double w : work) sum += w;
    return capture_fanout(g_main, order, stream_of, base, slot, key, sum / count, st,
                          [&](int i, cudaStream_t sk, char* sl) { return run(probs[i], sl, slot, sk); });
}

size_t batched_steps_ws(size_t slot) { return align_up(slot, 256) * n_streams() + 512; }

}  // namespace

extern "C" {

size_t lsq_batched_workspace_size(int32_t hpne, int32_t count, const lsq_batch_problem* probs) {
    if (count <= 0 || !probs) return 0;
    for (int i = 0; i < count; ++i)
        if (check_problem(probs[i]) != LSQ_OK) return 0;
    Plan P = make_plan(hpne != 0, count, probs);
    return P.head_bytes + P.slot_bytes * n_streams() + 512;
}

lsq_status lsq_pne_solve_batched(int32_t count, const lsq_batch_problem* probs, void* ws, size_t ws_bytes,
                                 void* stream) {
    return batched(false, count, probs, ws, ws_bytes, (cudaStream_t)stream);
}

lsq_status lsq_hpne_solve_batched(int32_t count, const lsq_batch_problem* probs, void* ws, size_t ws_bytes,
                                  void* stream) {
    return batched(true, count, probs, ws, ws_bytes, (cudaStream_t)stream);
}

size_t lsq_sketch_batched_workspace_size(int32_t count, const lsq_sketch_problem* probs) {
    if (count <= 0 || !probs) return 0;
    size_t slot = 0;
    for (int i = 0; i < count; ++i) {
        if (check_sketch_problem(probs[i]) != LSQ_OK) return 0;
        slot = std::max(slot, sketch_slot_bytes(probs[i]));
    }
    return batched_steps_ws(slot);
}

lsq_status lsq_sketch_batched(int32_t count, const lsq_sketch_problem* probs, void* ws, size_t ws_bytes,
                              void* stream) {
    return batched_steps(
        2, count, probs, ws, ws_bytes, (cudaStream_t)stream, check_sketch_problem, sketch_slot_bytes,
        [](const lsq_sketch_problem& p) { return 2.0 * (double)p.m * (double)p.n * (double)p.opts.s; },
        [](const lsq_sketch_problem& p, char* slot, size_t bytes, cudaStream_t sk) {
            return lsq_sketch(p.A, p.m, p.n, p.lda, &p.opts, p.As, p.ldas, p.colexp, p.info, slot, bytes, sk);
        });
}

size_t lsq_precond_qr_batched_workspace_size(int32_t count, const lsq_qr_problem* probs) {
    if (count <= 0 || !probs) return 0;
    size_t slot = 0;
    for (int i = 0; i < count; ++i) {
        if (check_qr_problem(probs[i]) != LSQ_OK) return 0;
        slot = std::max(slot, qr_slot_bytes(probs[i]));
    }
    return batched_steps_ws(slot);
}

lsq_status lsq_precond_qr_batched(int32_t count, const lsq_qr_problem* probs, void* ws, size_t ws_bytes,
                                  void* stream) {
    return batched_steps(
        3, count, probs, ws, ws_bytes, (cudaStream_t)stream, check_qr_problem, qr_slot_bytes,
        [](const lsq_qr_problem& p) { return 2.0 * (double)p.n * (double)p.n * (double)p.s; },
        [](const lsq_qr_problem& p, char* slot, size_t bytes, cudaStream_t sk) {
            return lsq_precond_qr(p.As, p.s, p.n, p.ldas, p.as_prec, p.qr_prec, p.colexp, p.Rs, p.ldr, p.info, slot,
                                  bytes, sk);
        });
}

}  // extern "C"
