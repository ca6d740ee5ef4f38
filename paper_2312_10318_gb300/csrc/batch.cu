// Batches: several lattices advanced together.  Per time step the members are
// grouped by (storage format, boundary flavour, G mode, parity of the current
// level) and each group is one specialised launch (lb_batch.cuh); runs of
// kGraphSteps steps are captured once into a CUDA graph and replayed.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <new>
#include <tuple>
#include <vector>

#include "lb_batch.cuh"
#include "lb_handle.h"

namespace {

constexpr int kGraphSteps = 32;  // steps per captured graph (even: parity and Phi
                                 // buffers return to their start after a replay)
constexpr size_t kMaxGraphs = 4;

}  // namespace

struct trtrlb_batch {
    cudaStream_t stream = nullptr;
    cudaStream_t copy_in = nullptr;    // uploads, downloads, and initial states and
    cudaStream_t copy_out = nullptr;   // moments, of trtrlb_batch_solve (created on
    cudaStream_t aux = nullptr;        // its first call)
    std::vector<trtrlb_t> lats;
    // runs of kGraphSteps steps, captured once per start (parity, Phi buffer and
    // population buffer of every member), at most kMaxGraphs of them
    std::map<std::vector<int>, cudaGraphExec_t> graphs;
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
}

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

int log2i(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
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

// Launches n steps of every member from the states `sim` (one per member),
// which it advances.  A member whose lattice the two-step kernel runs takes
// single steps to an odd level and for a last odd one, and two at a time
// between; members at different points share the launches they can.  closed: n
// is kGraphSteps and every member must end at the parity and on the buffers it
// began with, so that the launches can be replayed: every count of flips must
// be even, which 16 launches of two steps from an odd level are, and, from an
// even one, a single step, 14 launches of two and three single steps.
cudaError_t launch_steps(trtrlb_batch* b, std::vector<trt::State>& sim, int64_t n, bool closed = false) {
    using Key = std::tuple<int, int, int, int>;  // storage, flavour, g_mode, odd
    std::vector<int64_t> done(sim.size(), 0);
    std::vector<int64_t> last(sim.size(), n);    // no launch of two steps ends after it
    for (size_t i = 0; i < sim.size(); ++i)
        if (closed && sim[i].parity == 0) last[i] = n - 3;
    for (int64_t q = 0; q < n; ++q) {
        std::map<Key, std::vector<int>> groups;
        std::map<std::tuple<int, int>, std::vector<int>> pairs;   // storage, g_mode
        std::vector<int> tma, alone;
        for (int i = 0; i < (int)sim.size(); ++i) {
            if (done[i] != q) continue;
            const trtrlb_lattice* h = b->lats[i];
            const trt::State& s = sim[i];
            if (s.g_mode == TRTRLB_G_CURRENT) {
                // two-buffer members: the small TMA-fed ones share launches, the
                // others run one launch each
                (shares_tma_launch(h) ? tma : alone).push_back(i);
                done[i] += 1;
            } else if (s.pair && s.parity == 1 && q + 2 <= last[i]) {
                pairs[{h->p.storage, s.g_mode}].push_back(i);
                done[i] += 2;
            } else {
                const int flav = s.general ? trt::FLAV_GENERAL : (s.vec ? trt::FLAV_VECTOR : trt::FLAV_PERIODIC);
                groups[Key{h->p.storage, flav, s.g_mode, s.parity}].push_back(i);
                done[i] += 1;
            }
        }
        for (const auto& kv : pairs) {
            std::vector<const trt::State*> m;
            for (int i : kv.second) m.push_back(&sim[i]);
            const cudaError_t e = TRT_DISPATCH_S(std::get<0>(kv.first), step_pair(m.data(), (int)m.size(), b->stream));
            if (e != cudaSuccess) return e;
            for (int i : kv.second) trt::after_pair(sim[i]);
        }
        for (const auto& kv : groups) {
            const Key& k = kv.first;
            std::vector<const trt::State*> m;
            std::vector<int> cur, l2;
            for (int i : kv.second) {
                m.push_back(&sim[i]);
                cur.push_back(sim[i].cur);
                l2.push_back(log2i(b->lats[i]->tile_w));
            }
            cudaError_t e = TRT_DISPATCH_S(
                std::get<0>(k), step_group(m.data(), cur.data(), l2.data(), (int)m.size(),
                                           std::get<3>(k) != 0, std::get<1>(k),
                                           std::get<2>(k), b->stream));
            for (int i : kv.second) {
                if (e == cudaSuccess && sim[i].nghost > 0)
                    e = TRT_DISPATCH_S(std::get<0>(k), ghost_pass(sim[i], 0, b->stream));
                sim[i].parity ^= 1;
                if (sim[i].g_mode == TRTRLB_G_LAGGED) sim[i].cur ^= 1;
            }
            if (e != cudaSuccess) return e;
        }
        std::vector<const trt::State*> m;
        for (int i : tma) m.push_back(&sim[i]);
        if (!m.empty()) {
            const cudaError_t e = trt::Ops<float>::step_ab_group(m.data(), (int)m.size(), 0, b->stream);
            if (e != cudaSuccess) return e;
        }
        for (int i : alone) {
            const cudaError_t e = TRT_DISPATCH_S(b->lats[i]->p.storage, step_ab(sim[i], 0, b->stream));
            if (e != cudaSuccess) return e;
            tma.push_back(i);
        }
        for (int i : tma) {
            void* t = sim[i].f;
            sim[i].f = sim[i].f2;
            sim[i].f2 = t;
        }
    }
    return cudaSuccess;
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
    std::vector<trt::State> sim;
    for (trtrlb_lattice* h : b->lats) {
        trt::keep_spare(h);   // graphs name it
        sim.push_back(h->s);
    }
    int64_t done = 0;
    cudaError_t e = cudaSuccess;
    if (b->stream != nullptr && nsteps >= kGraphSteps) {
        // to odd levels, where the runs of two start, if that is a step for all
        bool odd_pair = false, even_pair = false;
        for (const trt::State& x : sim) (x.parity ? odd_pair : even_pair) |= x.pair;
        if (even_pair && !odd_pair && nsteps > kGraphSteps) {
            e = launch_steps(b, sim, 1);
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
    e = launch_steps(b, sim, nsteps - done);
    if (e != cudaSuccess) return cuda_fail(b, e, "batch step");
    for (size_t i = 0; i < sim.size(); ++i) {
        b->lats[i]->s = sim[i];
        b->lats[i]->t += nsteps;
    }
    return TRTRLB_OK;
}

const char* trtrlb_batch_last_error(trtrlb_batch_t b) { return b ? b->err : ""; }

}  // extern "C"
