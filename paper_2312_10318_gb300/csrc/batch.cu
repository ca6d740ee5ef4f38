// Batches: several lattices advanced together.  The members are grouped by
// (storage format, boundary flavour, G mode, parity of the current level) and
// each group takes one specialised launch per step (lb_batch.cuh) or two steps
// (lb_pair.cuh); runs of kGraphSteps steps are captured once into a CUDA graph
// and replayed.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <new>
#include <utility>
#include <vector>

#include "lb_batch.cuh"
#include "lb_handle.h"

namespace {

constexpr int kGraphSteps = 32;  // steps per captured graph (even: parity and Phi
                                 // buffers return to their start after a replay)
constexpr size_t kMaxGraphs = 4;
constexpr size_t kSideStreams = trt::kBatchStreams - 1;

}  // namespace

struct trtrlb_batch {
    cudaStream_t stream = nullptr;
    cudaStream_t copy_in = nullptr;    // uploads, downloads, and initial states and
    cudaStream_t copy_out = nullptr;   // moments, of trtrlb_batch_solve (created on
    cudaStream_t aux = nullptr;        // its first call)
    std::vector<cudaStream_t> side;    // classes of members beside the batch's stream
    std::vector<cudaEvent_t> joined;   // (created when first used)
    cudaEvent_t forked = nullptr;
    std::vector<trtrlb_t> lats;
    // runs of kGraphSteps steps, captured once per start (parity, Phi buffer and
    // population buffer of every member), at most kMaxGraphs of them
    std::map<std::vector<int>, cudaGraphExec_t> graphs;
    std::vector<SparePins*> held;      // the members' second buffers, while there are graphs
    char err[256] = "";
};

namespace {

int fail(trtrlb_batch* b, int code, const char* msg) {
    std::snprintf(b->err, sizeof b->err, "%s", msg);
    return code;
}

int cuda_fail(trtrlb_batch* b, cudaError_t e, const char* where) {
    std::snprintf(b->err, sizeof b->err, "%s: %s", where, cudaGetErrorString(e));
    return TRTRLB_ECUDA;
}

void drop_graphs(trtrlb_batch* b) {
    for (const auto& kv : b->graphs) cudaGraphExecDestroy(kv.second);
    b->graphs.clear();
    for (SparePins* x : b->held) x->unpin();
    b->held.clear();
}

// Pins the members' second buffers for the length of a call.
struct CallPins {
    std::vector<SparePins*> held;
    ~CallPins() {
        for (SparePins* x : held) x->unpin();
    }
    void add(SparePins* x) {
        held.push_back(x);
        x->pin();
    }
};

std::vector<int> signature(const trtrlb_batch* b, const std::vector<trt::State>& sim) {
    std::vector<int> sig;
    for (size_t i = 0; i < sim.size(); ++i) {
        sig.push_back(sim[i].parity);
        sig.push_back(sim[i].cur);
        sig.push_back(sim[i].f == b->lats[i]->f ? 0 : 1);   // two-buffer lattices alternate buffers
        sig.push_back(sim[i].pair ? 1 : 0);
    }
    return sig;
}

#define TRT_DISPATCH_S(storage, CALL)                                                 \
    [&]() -> cudaError_t {                                                            \
        switch (storage) {                                                            \
            case TRTRLB_F64: { using S = double; return trt::Ops<S>::CALL; }          \
            case TRTRLB_F64_DW: { using S = trt::f64dw; return trt::Ops<S>::CALL; }   \
            case TRTRLB_F32: { using S = float; return trt::Ops<S>::CALL; }           \
            case TRTRLB_F16_SHIFTED: { using S = __half; return trt::Ops<S>::CALL; }  \
            default: { using S = __nv_bfloat16; return trt::Ops<S>::CALL; }           \
        }                                                                             \
    }()

// Members that take the same launches: of one format, kernel, G mode and parity
// of the current level.  tma: the small TMA-fed two-buffer members, which share
// launches of single steps; the other two-buffer members take their own, and
// without launches of two steps are classes of their own.
struct Class {
    int storage, flavour, g_mode, parity;
    bool pair, tma;
    std::vector<int> members;
    long long nodes = 0;
};

std::vector<Class> classes_of(const trtrlb_batch* b, const std::vector<trt::State>& sim) {
    std::vector<Class> out;
    for (int i = 0; i < (int)sim.size(); ++i) {
        const trtrlb_lattice* h = b->lats[i];
        const trt::State& s = sim[i];
        const bool ab = s.g_mode == TRTRLB_G_CURRENT, tma = shares_tma_launch(h);
        const int flav = s.general ? trt::FLAV_GENERAL : (s.vec ? trt::FLAV_VECTOR : trt::FLAV_PERIODIC);
        Class* c = nullptr;
        for (Class& x : out)
            if (x.storage == h->p.storage && x.flavour == flav && x.g_mode == s.g_mode && x.parity == s.parity &&
                x.pair == s.pair && x.tma == tma && (!ab || tma || s.pair))
                c = &x;
        if (!c) {
            out.push_back(Class{h->p.storage, flav, s.g_mode, s.parity, s.pair, tma, {}, 0});
            c = &out.back();
        }
        c->members.push_back(i);
        c->nodes += (long long)s.nx * s.ny;
    }
    return out;
}

// Sets which members take launches of two steps in the states `sim` of a run: those
// that can, without those that the launches would not pay for: decided over those of one format, flavour and G mode,
// which share launches when their parities agree.  Only those that make up half of
// the batch: beside larger classes it is not the length of their launches that
// counts but their work, which two steps at a time have less of (21 served lattices
// of three formats, 49 steps: 4.57 ms, 4.73 with the small walled class in single
// steps).
void choose_two_steps(const trtrlb_batch* b, std::vector<trt::State>& sim, bool replayed) {
    std::vector<bool> seen(sim.size(), false);
    long long all = 0;
    for (size_t i = 0; i < sim.size(); ++i) {
        all += (long long)sim[i].nx * sim[i].ny;
        sim[i].pair = b->lats[i]->s.pair;
    }
    for (size_t i = 0; i < sim.size(); ++i) {
        if (seen[i] || !sim[i].pair) continue;
        std::vector<trtrlb_lattice*> m;
        std::vector<size_t> at;
        long long nodes = 0;
        for (size_t k = i; k < sim.size(); ++k) {
            const trt::State &x = sim[k], &y = sim[i];
            if (!x.pair || b->lats[k]->p.storage != b->lats[i]->p.storage || x.g_mode != y.g_mode ||
                x.general != y.general)
                continue;
            seen[k] = true;
            m.push_back(b->lats[k]);
            at.push_back(k);
            nodes += (long long)x.nx * x.ny;
        }
        if (2 * nodes < all || trt::run_pays(m.data(), (int)m.size(), replayed, true)) continue;
        for (size_t k : at) sim[k].pair = false;
    }
}

// n steps of the members of class c from the states `sim`, which it advances.
// Where the two-step kernel runs them: a single step to an odd level, two at a
// time, and single steps for the rest.  closed: the members end on the buffers
// that single steps would have left them at (trt::pair_launches); with n =
// kGraphSteps those are the ones they began on, and the launches can be replayed.
cudaError_t launch_class(trtrlb_batch* b, const Class& c, std::vector<trt::State>& sim, int64_t n, bool closed,
                         cudaStream_t st) {
    std::vector<const trt::State*> m;
    for (int i : c.members) m.push_back(&sim[i]);
    const int k = (int)m.size();
    int64_t pairs = trt::pair_launches(*m[0], n, closed);
    int parity = c.parity;
    for (int64_t q = 0; q < n;) {
        cudaError_t e;
        if (pairs > 0 && (parity == 1 || c.g_mode == TRTRLB_G_CURRENT)) {
            e = TRT_DISPATCH_S(c.storage, step_pair(m.data(), k, st));
            for (int i : c.members) trt::after_pair(sim[i]);
            --pairs;
            q += 2;
        } else if (c.g_mode == TRTRLB_G_CURRENT) {
            e = c.tma ? trt::Ops<float>::step_ab_group(m.data(), k, st)
                      : cudaSuccess;
            for (int i = 0; !c.tma && i < k && e == cudaSuccess; ++i)
                e = TRT_DISPATCH_S(c.storage, step_ab(*m[i], st));
            for (int i : c.members) std::swap(sim[i].f, sim[i].f2);
            q += 1;
        } else {
            e = TRT_DISPATCH_S(c.storage, step_group(m.data(), k, parity != 0, c.flavour, c.g_mode, st));
            for (int i : c.members) {
                if (e == cudaSuccess && sim[i].nghost > 0) e = TRT_DISPATCH_S(c.storage, ghost_pass(sim[i], st));
                sim[i].parity ^= 1;
                if (c.g_mode == TRTRLB_G_LAGGED) sim[i].cur ^= 1;
            }
            parity ^= 1;
            q += 1;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Launches n steps of every member from the states `sim` (one per member), which
// it advances.  The classes never read one another's lattices, so each takes all
// its steps on a stream of its own, forked from the batch's stream and joined to
// it (not from the default stream, which other work may expect to order with).
// Kernels that issue bounds (double-word) and kernels that memory bounds then
// share the SMs, and small classes run beside large ones: the 240 channels of
// three formats in 20.0 us per step (60 in line before, with 32-wide tiles).
cudaError_t launch_steps(trtrlb_batch* b, std::vector<trt::State>& sim, int64_t n, bool closed) {
    if (n == 0) return cudaSuccess;
    std::vector<Class> cs = classes_of(b, sim);
    if (b->stream == nullptr || cs.size() == 1) {
        for (const Class& c : cs) {
            const cudaError_t e = launch_class(b, c, sim, n, closed, b->stream);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    // the largest class on the batch's stream, the others beside it
    std::stable_sort(cs.begin(), cs.end(), [](const Class& x, const Class& y) { return x.nodes > y.nodes; });
    const size_t side = std::min(cs.size() - 1, kSideStreams);
    cudaError_t e = cudaSuccess;
    while (b->side.size() < side && e == cudaSuccess) {
        cudaStream_t x = nullptr;
        cudaEvent_t v = nullptr;
        e = cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&v, cudaEventDisableTiming);
        if (e == cudaSuccess) {
            b->side.push_back(x);
            b->joined.push_back(v);
        } else if (x) {
            cudaStreamDestroy(x);
        }
    }
    if (e == cudaSuccess && !b->forked) e = cudaEventCreateWithFlags(&b->forked, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(b->forked, b->stream);
    for (size_t k = 0; k < side && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->side[k], b->forked, 0);
    for (size_t k = 0; k < cs.size() && e == cudaSuccess; ++k)
        e = launch_class(b, cs[k], sim, n, closed, k % (side + 1) == 0 ? b->stream : b->side[k % (side + 1) - 1]);
    // join what was forked, whatever happened
    for (size_t k = 0; k < side && k < b->side.size(); ++k) {
        cudaError_t j = cudaEventRecord(b->joined[k], b->side[k]);
        if (j == cudaSuccess) j = cudaStreamWaitEvent(b->stream, b->joined[k], 0);
        if (e == cudaSuccess) e = j;
    }
    return e;
}

// The graph of kGraphSteps steps from `sim`, captured if it is not there yet.
int graph_from(trtrlb_batch* b, const std::vector<trt::State>& sim, cudaGraphExec_t* out) {
    const std::vector<int> sig = signature(b, sim);
    const auto it = b->graphs.find(sig);
    if (it != b->graphs.end()) {
        *out = it->second;
        return TRTRLB_OK;
    }
    if (b->graphs.size() >= kMaxGraphs) drop_graphs(b);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(b, e, "graph capture");
    std::vector<trt::State> copy = sim;
    const cudaError_t le = launch_steps(b, copy, kGraphSteps, true);
    e = cudaStreamEndCapture(b->stream, &g);
    if (le != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(b, le, "graph capture launch");
    }
    if (e != cudaSuccess) return cuda_fail(b, e, "graph capture end");
    cudaGraphExec_t x = nullptr;
    e = cudaGraphInstantiate(&x, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(b, e, "graph instantiate");
    b->graphs[sig] = x;
    if (b->held.empty())               // (pinned already for this call)
        for (trtrlb_lattice* h : b->lats) {
            b->held.push_back(h->pins);
            h->pins->pin();
        }
    *out = x;
    return TRTRLB_OK;
}

}  // namespace

extern "C" {

int trtrlb_batch_create(void* stream, trtrlb_batch_t* out) {
    if (!out) return TRTRLB_EINVAL;
    trtrlb_batch* b = new (std::nothrow) trtrlb_batch();
    if (!b) return TRTRLB_ENOMEM;
    b->stream = static_cast<cudaStream_t>(stream);
    *out = b;
    return TRTRLB_OK;
}

int trtrlb_batch_destroy(trtrlb_batch_t b) {
    if (!b) return TRTRLB_OK;
    cudaStreamSynchronize(b->stream);
    drop_graphs(b);
    if (b->copy_in) cudaStreamDestroy(b->copy_in);
    if (b->copy_out) cudaStreamDestroy(b->copy_out);
    if (b->aux) cudaStreamDestroy(b->aux);
    for (cudaStream_t x : b->side) cudaStreamDestroy(x);
    for (cudaEvent_t x : b->joined) cudaEventDestroy(x);
    if (b->forked) cudaEventDestroy(b->forked);
    delete b;
    return TRTRLB_OK;
}

int trtrlb_batch_set(trtrlb_batch_t b, const trtrlb_t* lattices, int count) {
    if (!b) return TRTRLB_EINVAL;
    b->err[0] = 0;
    if (count < 0 || (count > 0 && !lattices)) return fail(b, TRTRLB_EINVAL, "bad lattice list");
    std::vector<trtrlb_t> l(lattices, lattices + count);
    for (int q = 0; q < count; ++q) {
        if (!l[q]) return fail(b, TRTRLB_EINVAL, "null lattice in the list");
        for (int r = 0; r < q; ++r)
            if (l[r] == l[q]) return fail(b, TRTRLB_EINVAL, "a lattice appears twice");
    }
    drop_graphs(b);
    b->lats.swap(l);
    return TRTRLB_OK;
}

int trtrlb_batch_solve(trtrlb_batch_t b, const double* const* rho, const double* const* ux,
                       const double* const* uy, int64_t nsteps, double* const* rho_out,
                       double* const* ux_out, double* const* uy_out) {
    if (!b) return TRTRLB_EINVAL;
    b->err[0] = 0;
    cudaError_t e = cudaSuccess;
    if (!b->copy_in) e = cudaStreamCreateWithFlags(&b->copy_in, cudaStreamNonBlocking);
    if (e == cudaSuccess && !b->copy_out) e = cudaStreamCreateWithFlags(&b->copy_out, cudaStreamNonBlocking);
    if (e == cudaSuccess && !b->aux) {
        // the highest priority: its short, compute-bound kernels are scheduled
        // between the steps' blocks instead of after them
        int lo = 0, hi = 0;
        e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&b->aux, cudaStreamNonBlocking, hi);
    }
    if (e != cudaSuccess) return cuda_fail(b, e, "solve streams");
    return trt::solve_members(b->lats.data(), (int)b->lats.size(), b->stream, b->aux, b->copy_in, b->copy_out,
                              rho, ux, uy, nsteps, rho_out, ux_out, uy_out, b->err);
}

int trtrlb_batch_step(trtrlb_batch_t b, int64_t nsteps) {
    if (!b) return TRTRLB_EINVAL;
    b->err[0] = 0;
    if (nsteps < 0) return fail(b, TRTRLB_EINVAL, "nsteps must be >= 0");
    if (nsteps == 0 || b->lats.empty()) return TRTRLB_OK;
    bool capturing = false, closed = false;
    cudaError_t e = trt::capturing(b->stream, &capturing);
    if (e != cudaSuccess) return cuda_fail(b, e, "batch step");
    std::vector<trt::State> sim;
    CallPins pins;
    for (trtrlb_lattice* h : b->lats) {
        std::lock_guard<std::mutex> lk(h->spare_mu);
        pins.add(h->pins);
        h->captured = h->captured || capturing;
        closed = closed || h->captured;
        sim.push_back(h->s);
    }
    const bool graphs = b->stream != nullptr && nsteps >= kGraphSteps;
    choose_two_steps(b, sim, graphs || capturing);
    int64_t done = 0;
    if (graphs) {
        // to odd levels, where the runs of two start, if that is a step for all
        bool odd_pair = false, even_pair = false;
        for (const trt::State& x : sim)
            if (x.g_mode != TRTRLB_G_CURRENT) (x.parity ? odd_pair : even_pair) |= x.pair;
        if (even_pair && !odd_pair && nsteps > kGraphSteps) {
            e = launch_steps(b, sim, 1, closed);
            done = 1;
            if (e != cudaSuccess) return cuda_fail(b, e, "batch step");
        }
        cudaGraphExec_t graph = nullptr;
        if (int rc = graph_from(b, sim, &graph)) return rc;
        for (; done + kGraphSteps <= nsteps; done += kGraphSteps) {
            e = cudaGraphLaunch(graph, b->stream);
            if (e != cudaSuccess) return cuda_fail(b, e, "graph launch");
        }
    }
    choose_two_steps(b, sim, capturing);
    e = launch_steps(b, sim, nsteps - done, closed);
    if (e != cudaSuccess) return cuda_fail(b, e, "batch step");
    for (size_t i = 0; i < sim.size(); ++i) {
        sim[i].pair = b->lats[i]->s.pair;
        b->lats[i]->s = sim[i];
        b->lats[i]->t += nsteps;
    }
    return TRTRLB_OK;
}

const char* trtrlb_batch_last_error(trtrlb_batch_t b) { return b ? b->err : ""; }

}  // extern "C"
