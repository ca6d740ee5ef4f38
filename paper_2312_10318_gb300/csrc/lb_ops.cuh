// Host-side launchers of the device kernels, one instantiation per storage
// format (lb_ops_<fmt>.cu), so the formats compile in parallel.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace trt {

// Storage tag of FP64 populations with double-word FP32 arithmetic (lb_dw.cuh).
struct f64dw;

// Threads per block of the diagnostics reduction.
constexpr int DIAG_THREADS = 256;

// Kernel flavours of a lattice's step.
enum : int { FLAV_GENERAL = 0, FLAV_PERIODIC = 1, FLAV_VECTOR = 2 };

// Nodes per thread of the vectorised kernel: 16 bytes of FP64 / FP32
// storage, VEC16_NODES elements of 16-bit storage.
constexpr int VEC16_NODES = 4;
inline int vec_width(int storage_bytes) { return storage_bytes == 2 ? VEC16_NODES : 16 / storage_bytes; }

// Format-independent description of a lattice's device state.
// TMA-fed two-buffer kernel (lb_ab_tma.cuh): a tile of 32 x TMA_TH nodes, a
// thread owning TMA_TH / 8 of them (one per 8 rows), and its box x0-4 .. x0+35
// by y0-1 .. y0+TMA_TH, all 9 population planes, in one of TMA_STAGES
// shared-memory stages.
constexpr int TMA_TH = 8, TMA_STAGES = 2;
constexpr int TMA_BX = 40, TMA_BY = TMA_TH + 2, TMA_XOFF = 4;
// Polls of an mbarrier before a kernel's wait gives up (microseconds suffice
// for a tile copy; the limit only bounds a wait that would never end).
constexpr long long kDefaultWaitLimit = 1ll << 22;

// Two-step kernel (lb_pair.cuh): nodes of a row a warp updates, warps per CTA.
constexpr int PAIR_W = 60, PAIR_WARPS = 4;
constexpr int PAIR_AB_W = 56;   // with Phi at the current level
inline int pair_strips(int nx, int width = PAIR_W) { return (nx + width - 1) / width; }

struct State {
    void* f;              // populations, S[9][ny][pitch]
    void* f2;             // second buffer: of the two-buffer G_CURRENT kernel, or of
                          // the two-step kernel (else null)
    bool pair;            // the two-step kernel advances this lattice from odd levels
    const unsigned* pinfo;     // its maps of a general lattice (lb_pair.cuh): a word per node,
    const unsigned* pspecial;  // [ny][pitch], and a bit per strip and row, [strips][(ny + 31) / 32]
    int sms;              // multiprocessors of the device
    bool crowded;         // general: at least half of the row segments (seg) are not interior
    void* phi[2];         // Phi buffers, C[2][ny][pitch]
    int cur;              // phi[cur] holds the previous level
    const uint8_t* mask;  // device [ny][pitch] or nullptr
    const uint8_t* seg;   // general lattices: device [ny][segs], 1 where the 32-node row
                          // segment and all its neighbours are plain fluid (or nullptr)
    int segs;             // segments per row, (nx + 31) / 32
    const int* ghosts;    // device list of outlet ghost offsets
    int nghost;
    int nx, ny, pitch;
    long long plane;
    int px, py;
    bool general;         // walls, mask or non-periodic edges present
    bool vec;             // the vectorised kernel runs this lattice
    int col_h;            // G_CURRENT: rows per band of the column-walking two-buffer
                          // kernel, which runs the step; 0: another kernel
    int tile_w;           // scalar kernels: widest tile (narrow lattices and small launches
                          // take less: scalar_tile, scalar_threads)
    int g_mode;
    double tau1, tau2, gx, gy, rho0;
    double wall_ux, wall_uy, wall_rho;
    double outlet_rho;    // density of Zou-He pressure outlet nodes
    int parity;           // parity of the current level
    // FP32 periodic G_CURRENT lattices: TMA descriptors (CUtensorMap, host
    // memory) of the population buffers, tma_map[k] describing tma_buf[k]
    const void* tma_buf[2];
    const void* tma_map[2];
    int tma_grid;         // persistent grid of the TMA kernel (0: not used)
    int* kerr;            // device flag: a kernel's bounded wait ran out
    long long wait_limit; // polls before a kernel's wait gives up
};

template <typename S> struct Ops {
    // One time step (plus the outlet-ghost pass); flips parity and Phi buffers.
    static cudaError_t step(State& s, cudaStream_t st);
    // Two time steps of n lattices (State::pair, at an odd level, same flavour
    // and G mode) in one launch per GROUP_MAX of them; the caller swaps f and f2,
    // and with Phi lagged the Phi buffers.
    static cudaError_t step_pair(const State* const* members, int n, cudaStream_t st);
    // Fills a general lattice's maps of the two-step kernel.
    static cudaError_t pair_maps(const State& s, unsigned* info, unsigned* special, cudaStream_t st);
    static cudaError_t phi_static(State& s, cudaStream_t st);
    // *differ (device) := whether the Phi buffers of a lattice with a mask differ
    // at nodes whose Phi no step changes; formats of the two-step kernel only.
    static cudaError_t phi_static_differs(const State& s, int* differ, cudaStream_t st);
    static cudaError_t init(State& s, const double* rho, const double* ux, const double* uy,
                            cudaStream_t st);
    static cudaError_t moments(const State& s, double* rho, double* ux, double* uy,
                               cudaStream_t st);
    static cudaError_t get_f(const State& s, double* f, double* phi, cudaStream_t st);
    static cudaError_t set_f(State& s, const double* f, const double* phi, cudaStream_t st);
    // Deterministic FP64 diagnostics; part holds diag_blocks() * 8 doubles.
    static cudaError_t diagnostics(const State& s, double* part, double* out, cudaStream_t st);
    // One batched step of n lattices that share the kernel flavour (FLAV_*),
    // G mode and the parity of their current level (odd).
    static cudaError_t step_group(const State* const* members, int n, bool odd, int flavour, int g_mode,
                                  cudaStream_t st);
    // Outlet-ghost pass after a step from the state s (its parity and Phi
    // buffer before that step).
    static cudaError_t ghost_pass(const State& s, cudaStream_t st);
    // Two-buffer G_CURRENT step from s.f to s.f2; the caller swaps them.
    static cudaError_t step_ab(const State& s, cudaStream_t st);
    // Persistent grid (resident CTAs per SM x SMs) of the TMA-fed two-buffer
    // kernel on the current device; 0 for formats that do not have it.
    static int tma_grid();
    // Whether the TMA-fed two-buffer kernel advances this lattice (FP32,
    // periodic without a mask, G_CURRENT, descriptors present).
    static bool tma_eligible(const State& s);
    // Two-buffer step of n such lattices, up to 16 per launch.
    static cudaError_t step_ab_group(const State* const* members, int n, cudaStream_t st);
};

int diag_blocks(const State& s);

// FP64 comparison of velocity fields (compare.cu): blocks of the first level
// (as many as diag_blocks gives for the same node count) and the launcher.
// ux, uy, rx, ry are dense [ny][nx] device fields; mask is a lattice's pitched
// device mask or null; part holds compare_blocks(nx * ny) * 8 doubles; out
// receives TRTRLB_CMP_N doubles (include/trtrlb.h).
int compare_blocks(long long nodes);
cudaError_t compare_fields(const double* ux, const double* uy, const double* rx, const double* ry,
                           const uint8_t* mask, int nx, int ny, int pitch, int px, int py,
                           double* part, double* out, cudaStream_t st);

}  // namespace trt
