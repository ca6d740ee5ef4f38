// Internal layout of a lattice handle, shared by the C-ABI translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "lb_ops.cuh"
#include "lb_pair_rule.h"
#include "trtrlb.h"

// Who, beside the handle, names a lattice's second buffer: batches while a call or
// a captured graph of theirs does.  A batch may outlive its members, so this does
// too: refs counts the handle and the batches that hold it.
struct SparePins {
    std::atomic<int> refs{1}, pins{0};
    void unref() {
        if (--refs == 0) delete this;
    }
    void pin() { ++refs, ++pins; }
    void unpin() { --pins, unref(); }
};

// never (a kernel of single steps was chosen), in runs in which it pays
// (TRTRLB_KERNEL_AUTO: two_steps_pay), or always (trtrlb_set_two_step).
enum class TwoStep : unsigned char { OFF, AUTO, ALWAYS };

struct trtrlb_lattice {
    trtrlb_params p;
    trt::State s;
    cudaStream_t stream;
    int64_t t;           // steps since init / set_f
    void* f;             // device allocations owned by the handle
    void* f2;            // second population buffer (G_CURRENT; the two-step kernel's), or null
    void* phi;           // both Phi buffers in one allocation
    uint8_t* mask;
    uint8_t* seg;        // interior row segments of a general lattice (State::seg), or null
    unsigned* pair_map;  // State::pinfo and State::pspecial of a general lattice, or null
    int* ghosts;
    double* stage;       // FP64 staging for host transfers and comparisons
    int stage_fields;    // its size in fields of nx * ny doubles (3, 4 or 11)
    double* part;        // diagnostics partials (scratch)
    double* dout;        // result of diagnostics (8 doubles) and comparisons (TRTRLB_CMP_N)
    std::atomic<int64_t> bytes;   // (another thread's reclaim_spares lowers it)
    int tile_w;          // scalar-kernel tile width in the batched path (32 .. 256 nodes)
    int variant;         // TRTRLB_KERNEL_AUTO / SCALAR / VECTOR / COLUMN
    TwoStep two_step;    // two steps per launch where the lattice allows it
    void* tmaps;         // two CUtensorMap (host) of the FP32 periodic G_CURRENT kernel, or null
    int* kerr;           // device flag set when a kernel's bounded wait ran out, or null
    int tma_grid;        // persistent grid of the TMA kernel on this device (0: none)
    int sms;             // multiprocessors of the handle's device
    // Another thread's failed allocation may give back f2 of a lagged lattice
    // (reclaim_spares): held there, and by every call that reads or writes f2, s.f2
    // or s.pair after create.
    std::mutex spare_mu;
    bool phi_given;      // the Phi buffers may differ at nodes whose Phi no step changes
    SparePins* pins;     // f2 is not given back while something pins it
    bool captured;       // nor ever, once a caller's graph holds steps of it (trt::pair_launches)
    char err[256];
};

// Lattices below this many nodes share the TMA-fed two-buffer launches of a
// batch (one persistent grid, one tail: 3 x 1024^2 FP32 54.2 -> 56.6 GLUPS);
// larger ones take a launch each (one 4096^2 lattice steps alone in 0.231 ms,
// three of them sharing a launch in 0.90 ms).
constexpr long long kTmaShareMaxNodes = 2048ll * 2048ll;

inline bool shares_tma_launch(const trtrlb_lattice* h) {
    return h->s.g_mode == TRTRLB_G_CURRENT && h->p.storage == TRTRLB_F32 &&
           trt::Ops<float>::tma_eligible(h->s) && (long long)h->p.nx * h->p.ny < kTmaShareMaxNodes;
}

namespace trt {
constexpr int kTmaShare = 16;     // lattices per shared TMA-fed launch
constexpr int kBatchStreams = 6;  // a batch's own stream and those beside it

// Adds lattice h, at state s, to the run r that it would share launches in (r of
// n - 1 such lattices before: {} for n = 1).
inline void add_to_run(PairRun& r, const trtrlb_lattice* h, int n, bool replayed, bool batch) {
    const State& s = h->s;
    r.current = s.g_mode == TRTRLB_G_CURRENT;
    r.off = s.g_mode == TRTRLB_G_OFF;
    const int width = r.current ? PAIR_AB_W : PAIR_W, together = shares_tma_launch(h) ? kTmaShare : kBatchStreams;
    r.members = n;
    r.nodes += (long long)s.nx * s.ny;
    r.columns += (long long)pair_strips(s.nx, width) * width * s.ny;
    r.tiled += (long long)(s.nx + 31) / 32 * 32 * s.ny;
    r.elem = h->p.storage == TRTRLB_F32 ? 4 : 2;
    r.general = s.general;
    r.ghosts = r.ghosts || s.nghost > 0;
    r.crowded = (n == 1 || r.crowded) && s.crowded;
    r.mask = r.mask || s.mask != nullptr;
    r.padded += s.plane;
    r.depth = (n + together - 1) / together;
    r.replayed = replayed;
    r.batch = batch;
}

// Whether st is being captured into a caller's graph.
inline cudaError_t capturing(cudaStream_t st, bool* on) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cs);
    *on = cs != cudaStreamCaptureStatusNone;
    return e;
}

// Launches of two steps in a run of n steps of a lattice that takes them (the
// other steps are single ones): from odd levels with Phi lagged or no G, so that
// a run from an even one begins with a single step, from any level with Phi at
// the current one.  Each swaps the population buffers, and with Phi lagged the
// Phi buffers once for two steps.  even: an even number of them, after which the
// lattice is at the parity and on the buffers that single steps would have left
// it at; graphs that are replayed need that, and so does every run of a lattice
// that a caller's graph names.
inline int64_t pair_launches(const State& s, int64_t n, bool even) {
    if (!s.pair) return 0;
    const int64_t first = s.g_mode != TRTRLB_G_CURRENT && s.parity == 0 ? 1 : 0;
    const int64_t k = n > first ? (n - first) / 2 : 0;
    return even ? k & ~(int64_t)1 : k;
}

// Whether a run of the n lattices h, all of one format, flavour and G mode and all
// able to, takes two steps per launch.
bool run_pays(trtrlb_lattice* const* h, int n, bool replayed, bool batch);

// Advances h by n time steps on st: two at a time from odd levels where the
// two-step kernel runs the lattice.
cudaError_t advance(trtrlb_lattice* h, int64_t n, cudaStream_t st);

// The effect of one launch of the two-step kernel on a lattice's state.
inline void after_pair(State& s) {
    void* t = s.f;
    s.f = s.f2;
    s.f2 = t;
    if (s.g_mode == TRTRLB_G_LAGGED) s.cur ^= 1;
}

// Body of trtrlb_batch_solve over the members m[0 .. count): see trtrlb.h.
// st runs the members' steps, aux their initial states and moments; cin and
// cout their uploads and downloads.
int solve_members(trtrlb_lattice* const* m, int count, cudaStream_t st, cudaStream_t aux, cudaStream_t cin,
                  cudaStream_t cout, const double* const* rho, const double* const* ux, const double* const* uy,
                  int64_t nsteps, double* const* rho_out, double* const* ux_out, double* const* uy_out,
                  char* err);
}  // namespace trt
