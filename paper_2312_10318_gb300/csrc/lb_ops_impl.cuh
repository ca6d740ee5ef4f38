// Definitions of Ops<S> (lb_ops.cuh); included once per storage format.
#pragma once
#include <type_traits>

#include "lb_ab.cuh"
#include "lb_ab_col.cuh"
#include "lb_ab_tma.cuh"
#include "lb_aux.cuh"
#include "lb_batch.cuh"
#include "lb_ops.cuh"
#include "lb_pair.cuh"

namespace trt {

template <typename C>
static Args<C> make_args(const State& s, bool swap_phi = false) {
    Args<C> a;
    a.f = s.f;
    const int in = swap_phi ? 1 - s.cur : s.cur;
    a.phi_in = static_cast<const C*>(s.phi[in]);
    a.phi_out = static_cast<C*>(s.phi[1 - in]);
    a.mask = s.mask;
    a.seg = s.seg;
    a.segs = s.segs;
    a.nx = s.nx; a.ny = s.ny; a.pitch = s.pitch; a.plane = s.plane;
    a.px = s.px; a.py = s.py;
    const double k1 = 1.0 - 1.0 / s.tau1, k2 = 1.0 - 1.0 / s.tau2;
    a.k1 = (C)k1;
    a.k1lo = (C)(k1 - (double)a.k1);   // 0 when C is double
    a.k2 = (C)k2;
    a.k2lo = (C)(k2 - (double)a.k2);
    a.kf = (C)(1.0 - 1.0 / (2.0 * s.tau1));
    a.gx = (C)s.gx; a.gy = (C)s.gy; a.rho0 = (C)s.rho0;
    a.hgx = (C)(0.5 * s.gx); a.hgy = (C)(0.5 * s.gy);
    for (int i = 0; i < 9; ++i) {
        // 2 w_i rho_w (e_i.u_w) / c_s^2, subtracted from f*_i when e_i points
        // into a moving wall (Ladd's correction)
        const double eu = ex(i) * s.wall_ux + ey(i) * s.wall_uy;
        a.corr[i] = (C)(6.0 * wgt(i) * s.wall_rho * eu);
    }
    a.phin_x = (C)(s.wall_rho * s.wall_ux * s.wall_ux * s.wall_ux);
    a.phin_y = (C)(s.wall_rho * s.wall_uy * s.wall_uy * s.wall_uy);
    a.zh_dr = (C)(s.rho0 - s.outlet_rho);
    return a;
}

static inline dim3 grid2d(const State& s, dim3 b) {
    return dim3((s.nx + b.x - 1) / b.x, (s.ny + b.y - 1) / b.y);
}

// Launches a step kernel (one that begins with chain_begin()) so that its set-up
// overlaps the end of the previous kernel of the stream.  Us per step without /
// with: FP64 64^2 6.2 / 4.1, FP32 250 x 246 3.1 / 2.2, 1024^2 10.2 / 8.7, 4096^2
// within noise.  Captured launches keep full edges, which a replay runs faster
// (240 channels, 256 steps: 5.1 ms, with programmatic edges 6.6).
template <typename P, typename... A>
static cudaError_t launch_chained(void (*kernel)(P, A...), dim3 g, dim3 b, cudaStream_t st, const P& p, A... rest) {
    cudaLaunchConfig_t c = {};
    c.gridDim = g;
    c.blockDim = b;
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cs);
    c.attrs = at;
    c.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;
    void* args[] = {const_cast<P*>(&p), &rest...};
    return cudaLaunchKernelExC(&c, reinterpret_cast<const void*>(kernel), args);
}

// Scalar kernels: threads per CTA of a launch over n lattices, and the tile width
// (a power of two) of one of them.  A lattice narrower than its tile takes the
// next power of two of its width, so that a warp spans rows instead of idling
// lanes (8-wide channels ran on a quarter of theirs, and FP64's pipe is busy for
// all 32).  A launch that would leave SMs without a CTA halves its CTAs, down to
// a warp: FP64 64^2 in 16 CTAs used 16 SMs' FP64 pipes.
// least: the narrowest tile.  With walls a warp of several rows runs the code of
// plain rows and that of rows at walls one after the other, so as long as every
// warp of one row has an SM quarter to itself, where idle lanes cost nothing, they
// stay that wide (us per step, replayed, tiles of 8 / 32: one channel of 8 x 256
// double-word 6.0 / 4.2, BF16 3.3 / 2.7, FP64 9.1 / 5.9; 16 of them 6.3 / 8.1, 4.0 / 4.0,
// 13.3 / 30.2).
static inline int least_tile(const State* const* m, int n) {
    long long warps = 0;
    for (int q = 0; q < n; ++q) warps += (long long)((m[q]->nx + 31) / 32) * m[q]->ny;
    return m[0]->general && warps <= 4ll * m[0]->sms ? 32 : 1;
}
static inline int scalar_tile(const State& s, int threads, int least) {
    int tw = s.tile_w > 0 ? s.tile_w : 128;
    while (tw > threads || (tw > least && tw / 2 >= s.nx)) tw /= 2;
    return tw;
}
// With a mask only FP64 halves them: a node's accesses depend on its neighbours'
// classes, which a CTA of several rows finds in its SM's L1 (us per step, replayed,
// CTAs of 256 / down to a warp: 128^2 with an obstacle FP32 3.4 / 4.0, double-word
// 4.6 / 5.6, FP64, whose pipe counts, 9.4 / 7.4).
static inline bool halves_ctas(const State* const* m, int n, bool fp64) {
    bool masks = false;
    for (int q = 0; q < n; ++q) masks = masks || m[q]->mask != nullptr;
    return fp64 || !masks;
}
static inline int scalar_threads(const State* const* m, int n, int rows, int most, int least, bool fp64) {
    int t = most;
    for (const int floor = halves_ctas(m, n, fp64) ? 32 : most; t > floor; t /= 2) {
        long long tiles = 0;
        for (int q = 0; q < n; ++q) {
            const int tw = scalar_tile(*m[q], t, least), th = t / tw * rows;
            tiles += (long long)((m[q]->nx + tw - 1) / tw) * ((m[q]->ny + th - 1) / th);
        }
        if (tiles >= 2 * m[0]->sms) break;
    }
    return t;
}

// Whether a launch's CTAs are all resident at 4 of 256 threads per SM
// (step_min_blocks).
static inline bool few_ctas(long long ctas, int threads, int sms) { return ctas * threads <= 4ll * 256 * sms; }

// Nodes per thread: the periodic double-word step takes two (thread_step), unless a
// launch has too few nodes to fill the SMs with them (two_rows).  With
// walls and masks it takes one: a segment at them steps its nodes one after the
// other, which all but the largest launches wait for at their end (us per step, one
// / two: channel 1024^2 49.4 / 54.9, 2048^2 178 / 169; periodic 4096^2 615 / 539),
// and the kernels that hold both forms took five minutes to compile.
template <typename S, bool GENERAL>
constexpr int rows_of_step() { return std::is_same<S, f64dw>::value && !GENERAL ? 2 : 1; }

// Whether a launch of the periodic double-word step takes two nodes per thread: from
// 512 nodes per SM on, 8 warps of two.  Below, a launch is as long as one thread's
// work (us per step, replayed, one / two: 64^2 3.0 / 3.7, 256^2 4.0 / 4.3, 320^2 6.7 /
// 6.7, 512^2 10.9 / 10.4, 16 lattices of 64^2 4.2 / 4.4, 8 of 128^2 6.9 / 6.8).
static inline bool two_rows(const State* const* m, int n) {
    long long nodes = 0;
    for (int q = 0; q < n; ++q) nodes += (long long)m[q]->nx * m[q]->ny;
    return nodes > 512ll * m[0]->sms;
}

template <typename S, bool ODD, bool GENERAL, int ROWS>
static void launch_scalar(const State& s, const Args<typename Fmt<S>::C>& a, cudaStream_t st) {
    const State* one = &s;
    if constexpr (ROWS == 2)
        if (!two_rows(&one, 1)) return launch_scalar<S, ODD, GENERAL, 1>(s, a, st);
    const int least = least_tile(&one, 1);
    const int t = scalar_threads(&one, 1, ROWS, step_threads<ROWS>(), least, std::is_same<S, double>::value),
              tw = scalar_tile(s, t, least);
    const dim3 b(tw, t / tw), g = grid2d(s, dim3(tw, t / tw * ROWS));
    if constexpr (few_variant<S, GENERAL>()) {
        if (few_ctas((long long)g.x * g.y, t, s.sms)) {
            if (s.g_mode == G_OFF) launch_chained(k_step<S, ODD, GENERAL, G_OFF, ROWS, true>, g, b, st, a);
            else launch_chained(k_step<S, ODD, GENERAL, G_LAGGED, ROWS, true>, g, b, st, a);
            return;
        }
    }
    if (s.g_mode == G_OFF) launch_chained(k_step<S, ODD, GENERAL, G_OFF, ROWS, false>, g, b, st, a);
    else launch_chained(k_step<S, ODD, GENERAL, G_LAGGED, ROWS, false>, g, b, st, a);
}

template <typename S, bool ODD>
static void launch_step(const State& s, const Args<typename Fmt<S>::C>& a, cudaStream_t st) {
    if (s.general) launch_scalar<S, ODD, true, rows_of_step<S, true>()>(s, a, st);
    else launch_scalar<S, ODD, false, rows_of_step<S, false>()>(s, a, st);
}

template <typename S, bool ODD>
static void launch_step_vec(const State& s, const Args<typename Fmt<S>::C>& a, cudaStream_t st) {
    constexpr int V = Pk<S>::V;
    const int spr = (s.nx + 32 * V - 1) / (32 * V);
    const long long nseg = (long long)spr * s.ny;
    const int blocks = (int)((nseg + 7) / 8);
    if (s.g_mode == G_OFF) launch_chained(k_step_vec<S, ODD, G_OFF>, blocks, 256, st, a, spr);
    else launch_chained(k_step_vec<S, ODD, G_LAGGED>, blocks, 256, st, a, spr);
}

template <typename S>
cudaError_t Ops<S>::step_ab(const State& s, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    if constexpr (std::is_same<S, float>::value) {
        if (tma_eligible(s)) {
            const State* one = &s;
            return step_ab_group(&one, 1, st);
        }
    }
    const Args<C> a = make_args<C>(s);
    if constexpr (!std::is_same<S, f64dw>::value) {
        if (s.col_h > 0 && !s.general) {
            const int gx = (s.nx + COL_W - 1) / COL_W, bands = (s.ny + s.col_h - 1) / s.col_h;
            const long long warps = (long long)gx * bands;
            const int blocks = (int)((warps + COL_WARPS - 1) / COL_WARPS);
            k_step_ab_col<S><<<blocks, COL_WARPS * 32, 0, st>>>(a, static_cast<S*>(s.f2), gx, bands, s.col_h);
            return cudaGetLastError();
        }
    }
    const dim3 g((s.nx + AB_TX - 1) / AB_TX, (s.ny + AB_TY - 1) / AB_TY);
    if (s.general) k_step_ab<S, true><<<g, AB_TX * AB_TY, 0, st>>>(a, static_cast<S*>(s.f2), 0);
    else k_step_ab<S, false><<<g, AB_TX * AB_TY, 0, st>>>(a, static_cast<S*>(s.f2), 0);
    return cudaGetLastError();
}

// Dynamic shared memory and carveout of a TMA kernel; occ becomes the smaller
// of its value and the kernel's resident CTAs per SM.
template <typename K>
static cudaError_t tma_setup(K kernel, int& occ) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TMA_SMEM_BYTES);
    // all of the unified L1/shared array as shared memory, so that the resident
    // CTAs the occupancy query counts are the ones that run (the grid is
    // persistent: one missing CTA per SM is a second wave)
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    int o = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kernel, AB_TX * AB_TY, TMA_SMEM_BYTES);
    if (e == cudaSuccess) occ = occ == 0 || o < occ ? o : occ;
    return e;
}

template <typename S>
bool Ops<S>::tma_eligible(const State& s) {
    return std::is_same<S, float>::value && !s.general && s.g_mode == G_CURRENT && s.tma_grid > 0 &&
           s.kerr != nullptr;
}

// Member k of a TMA launch; returns its tile count.
template <int MAXL>
static int tma_member(TmaGroup<MAXL>& g, int k, const State& s) {
    const int buf = s.f == s.tma_buf[0] ? 0 : 1;
    g.map[k] = *static_cast<const CUtensorMap*>(s.tma_map[buf]);
    g.a[k] = make_args<float>(s);
    g.dst[k] = static_cast<float*>(s.f2);
    g.err[k] = s.kerr;
    g.tiles_x[k] = (s.nx + AB_TX - 1) / AB_TX;
    return g.tiles_x[k] * ((s.ny + TMA_TH - 1) / TMA_TH);
}

template <int MAXL>
static cudaError_t launch_tma(const State* const* m, int n, cudaStream_t st) {
    TmaGroup<MAXL> g;
    g.n = n;
    g.tile_begin[0] = 0;
    int grid = 0;
    long long wait = 0;
    for (int k = 0; k < n; ++k) {
        g.tile_begin[k + 1] = g.tile_begin[k] + tma_member(g, k, *m[k]);
        grid = k == 0 || m[k]->tma_grid < grid ? m[k]->tma_grid : grid;
        wait = k == 0 || m[k]->wait_limit < wait ? m[k]->wait_limit : wait;
    }
    const int ntiles = g.tile_begin[n];
    if (ntiles == 0) return cudaSuccess;
    k_step_ab_tma<MAXL><<<ntiles < grid ? ntiles : grid, AB_TX * AB_TY, TMA_SMEM_BYTES, st>>>(g, ntiles, wait);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::step_ab_group(const State* const* members, int n, cudaStream_t st) {
    if constexpr (std::is_same<S, float>::value) {
        for (int k = 0; k < n; ++k)
            if (!tma_eligible(*members[k])) return cudaErrorInvalidValue;
        if (n == 1) return launch_tma<1>(members, 1, st);
        for (int k0 = 0; k0 < n; k0 += TMA_GROUP_MAX) {
            const int c = n - k0 < TMA_GROUP_MAX ? n - k0 : TMA_GROUP_MAX;
            const cudaError_t e = launch_tma<TMA_GROUP_MAX>(members + k0, c, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    } else {
        (void)members; (void)n; (void)st;
        return cudaErrorInvalidValue;
    }
}

template <typename S>
int Ops<S>::tma_grid() {
    if constexpr (std::is_same<S, float>::value) {
        int dev = 0, sms = 0, occ = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            tma_setup(k_step_ab_tma<1>, occ) != cudaSuccess ||
            tma_setup(k_step_ab_tma<TMA_GROUP_MAX>, occ) != cudaSuccess)
            return 0;
        return occ * sms;
    } else {
        return 0;
    }
}

template <typename S>
cudaError_t Ops<S>::step(State& s, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    if (s.g_mode == G_CURRENT) {
        const cudaError_t e = step_ab(s, st);
        void* t = s.f;
        s.f = s.f2;
        s.f2 = t;
        return e;
    }
    const Args<C> a = make_args<C>(s);
    if (s.vec) {
        if (s.parity == 0) launch_step_vec<S, false>(s, a, st);
        else launch_step_vec<S, true>(s, a, st);
    } else if (s.parity == 0) {
        launch_step<S, false>(s, a, st);
    } else {
        launch_step<S, true>(s, a, st);
    }
    if (s.nghost > 0) {
        const int t = 128, g = (s.nghost + t - 1) / t;
        if (s.parity == 0) launch_chained(k_ghosts<S, true>, g, t, st, a, s.ghosts, s.nghost);
        else launch_chained(k_ghosts<S, false>, g, t, st, a, s.ghosts, s.nghost);
    }
    s.parity ^= 1;
    if (s.g_mode == G_LAGGED) s.cur ^= 1;
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::phi_static(State& s, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    cudaError_t e = cudaMemsetAsync(s.phi[0], 0, sizeof(C) * 2 * s.plane, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.phi[1], 0, sizeof(C) * 2 * s.plane, st);
    if (e != cudaSuccess) return e;
    if (!s.mask) return cudaSuccess;
    const dim3 b(32, 8);
    const C inx = (C)(s.wall_rho * s.wall_ux * s.wall_ux * s.wall_ux);
    const C iny = (C)(s.wall_rho * s.wall_uy * s.wall_uy * s.wall_uy);
    k_phi_static<C><<<grid2d(s, b), b, 0, st>>>(s.mask, s.nx, s.ny, s.pitch, s.plane,
                                                static_cast<C*>(s.phi[0]),
                                                static_cast<C*>(s.phi[1]), inx, iny);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::phi_static_differs(const State& s, int* differ, cudaStream_t st) {
    if constexpr (sizeof(S) <= 4) {
        const cudaError_t e = cudaMemsetAsync(differ, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
        const dim3 b(32, 8);
        k_phi_static_differs<<<grid2d(s, b), b, 0, st>>>(s.mask, s.nx, s.ny, s.pitch, s.plane,
                                                         static_cast<const float*>(s.phi[0]),
                                                         static_cast<const float*>(s.phi[1]), differ);
        return cudaGetLastError();
    } else {
        (void)s; (void)differ; (void)st;
        return cudaErrorInvalidValue;
    }
}

template <typename S>
cudaError_t Ops<S>::init(State& s, const double* rho, const double* ux, const double* uy,
                         cudaStream_t st) {
    using C = typename Fmt<S>::C;
    s.parity = 0;
    s.cur = 0;
    const Args<C> a = make_args<C>(s, /*swap_phi=*/true);  // phi_out = phi[0] (the "in" level)
    const dim3 b(32, 8);
    k_init<S><<<grid2d(s, b), b, 0, st>>>(a, rho, ux, uy, s.rho0, s.gx, s.gy,
                                          static_cast<C*>(s.phi[1]));
    if (s.nghost > 0) {
        const int t = 128, g = (s.nghost + t - 1) / t;
        for (int q = 0; q < 2; ++q)
            k_ghost_phi<C><<<g, t, 0, st>>>(s.ghosts, s.nghost, s.nx, s.pitch, s.plane,
                                            static_cast<C*>(s.phi[q]));
    }
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::moments(const State& s, double* rho, double* ux, double* uy,
                            cudaStream_t st) {
    using C = typename Fmt<S>::C;
    const Args<C> a = make_args<C>(s);
    const dim3 b(32, 8);
    if (s.parity) k_moments<S, true><<<grid2d(s, b), b, 0, st>>>(a, rho, ux, uy);
    else k_moments<S, false><<<grid2d(s, b), b, 0, st>>>(a, rho, ux, uy);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::get_f(const State& s, double* f, double* phi, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    const Args<C> a = make_args<C>(s);
    const dim3 b(32, 8);
    if (s.parity) k_get_f<S, true><<<grid2d(s, b), b, 0, st>>>(a, f, phi);
    else k_get_f<S, false><<<grid2d(s, b), b, 0, st>>>(a, f, phi);
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::set_f(State& s, const double* f, const double* phi, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    s.parity = 0;
    const Args<C> a = make_args<C>(s);
    const dim3 b(32, 8);
    k_set_f<S><<<grid2d(s, b), b, 0, st>>>(a, f, phi);
    if (!phi) {
        k_phi_of_state<S><<<grid2d(s, b), b, 0, st>>>(a);
        if (s.nghost > 0) {
            const int t = 128, g = (s.nghost + t - 1) / t;
            k_ghost_phi<C><<<g, t, 0, st>>>(s.ghosts, s.nghost, s.nx, s.pitch, s.plane,
                                            static_cast<C*>(s.phi[s.cur]));
        }
    }
    return cudaGetLastError();
}

template <typename S>
cudaError_t Ops<S>::diagnostics(const State& s, double* part, double* out, cudaStream_t st) {
    using C = typename Fmt<S>::C;
    const Args<C> a = make_args<C>(s);
    const int nb = diag_blocks(s);
    if (s.parity) k_diag_partial<S, true><<<nb, DIAG_THREADS, 0, st>>>(a, part);
    else k_diag_partial<S, false><<<nb, DIAG_THREADS, 0, st>>>(a, part);
    k_diag_final<<<1, DIAG_THREADS, 0, st>>>(part, nb, out);
    return cudaGetLastError();
}

// FLAV: FLAV_GENERAL, FLAV_PERIODIC (scalar kernels) or FLAV_VECTOR.
template <typename S, bool ODD, int FLAV, int GMODE, int ROWS, int MAXL>
static cudaError_t launch_group(const State* const* m, int n, cudaStream_t st) {
    if constexpr (ROWS == 2 && FLAV == FLAV_PERIODIC)
        if (!two_rows(m, n)) return launch_group<S, ODD, FLAV, GMODE, 1, MAXL>(m, n, st);
    using C = typename Fmt<S>::C;
    constexpr int V = Pk<S>::V;
    GroupParams<C, MAXL> p;
    p.n = n;
    int tiles = 0;
    const int least = least_tile(m, n);
    const int threads = FLAV == FLAV_VECTOR
                            ? BATCH_THREADS
                            : scalar_threads(m, n, ROWS, step_threads<ROWS>(), least, std::is_same<S, double>::value);
    p.log2_threads = 0;
    while ((1 << p.log2_threads) < threads) ++p.log2_threads;
    for (int q = 0; q < n; ++q) {
        const State& v = *m[q];
        p.a[q] = make_args<C>(v);
        p.tile_begin[q] = tiles;
        if (FLAV == FLAV_VECTOR) {
            p.segs[q] = (v.nx + 32 * V - 1) / (32 * V);
            p.inv_d[q] = 1.0f / (float)p.segs[q];
            p.tiles_x[q] = 0;
            p.log2_tw[q] = 0;
            tiles += (int)(((long long)p.segs[q] * v.ny + 7) / 8);
        } else {
            const int tw = scalar_tile(v, threads, least), th = threads / tw * ROWS;
            p.log2_tw[q] = 0;
            while ((1 << p.log2_tw[q]) < tw) ++p.log2_tw[q];
            p.segs[q] = 0;
            p.tiles_x[q] = (v.nx + tw - 1) / tw;
            p.inv_d[q] = 1.0f / (float)p.tiles_x[q];
            tiles += p.tiles_x[q] * ((v.ny + th - 1) / th);
        }
    }
    p.tile_begin[n] = tiles;
    if (FLAV == FLAV_VECTOR)
        return launch_chained(k_step_group_vec<S, ODD, GMODE, MAXL>, tiles, BATCH_THREADS, st, p);
    else {
        constexpr bool GENERAL = FLAV == FLAV_GENERAL;
        if constexpr (few_variant<S, GENERAL>())
            if (few_ctas(tiles, threads, m[0]->sms))
                return launch_chained(k_step_group<S, ODD, GENERAL, GMODE, ROWS, true, MAXL>, tiles, threads, st, p);
        return launch_chained(k_step_group<S, ODD, GENERAL, GMODE, ROWS, false, MAXL>, tiles, threads, st, p);
    }
}

template <typename S, bool ODD, int FLAV, int GMODE>
static cudaError_t launch_group_sized(const State* const* m, int n, cudaStream_t st) {
    constexpr int ROWS = rows_of_step<S, FLAV == FLAV_GENERAL>();
    for (int q0 = 0; q0 < n; q0 += GROUP_MAX) {
        const int c = n - q0 < GROUP_MAX ? n - q0 : GROUP_MAX;
        cudaError_t e;
        // the double-word kernels, the longest to compile and to run, have one size
        if constexpr (std::is_same<S, f64dw>::value)
            e = launch_group<S, ODD, FLAV, GMODE, ROWS, GROUP_MAX>(m + q0, c, st);
        else
            e = c <= 4 ? launch_group<S, ODD, FLAV, GMODE, ROWS, 4>(m + q0, c, st)
                       : launch_group<S, ODD, FLAV, GMODE, ROWS, GROUP_MAX>(m + q0, c, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename S, bool ODD, int FLAV>
static cudaError_t launch_group_g(const State* const* m, int n, int g_mode, cudaStream_t st) {
    return g_mode == G_OFF ? launch_group_sized<S, ODD, FLAV, G_OFF>(m, n, st)
                           : launch_group_sized<S, ODD, FLAV, G_LAGGED>(m, n, st);
}

template <typename S>
cudaError_t Ops<S>::step_group(const State* const* m, int n, bool odd, int flavour, int g_mode, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (odd) {
        if (flavour == FLAV_GENERAL) return launch_group_g<S, true, FLAV_GENERAL>(m, n, g_mode, st);
        if (flavour == FLAV_VECTOR) return launch_group_g<S, true, FLAV_VECTOR>(m, n, g_mode, st);
        return launch_group_g<S, true, FLAV_PERIODIC>(m, n, g_mode, st);
    }
    if (flavour == FLAV_GENERAL) return launch_group_g<S, false, FLAV_GENERAL>(m, n, g_mode, st);
    if (flavour == FLAV_VECTOR) return launch_group_g<S, false, FLAV_VECTOR>(m, n, g_mode, st);
    return launch_group_g<S, false, FLAV_PERIODIC>(m, n, g_mode, st);
}

template <typename S, bool GENERAL, int GMODE, int MAXL>
static cudaError_t launch_pair(const State* const* m, int n, cudaStream_t st) {
    PairParams<MAXL> p;
    p.n = n;
    // general lattices leave a sixteenth of the slots to the parts of split tiles
    constexpr bool ab = GMODE == G_CURRENT;
    constexpr int width = ab ? PAIR_AB_W : PAIR_W;
    const long long slots = (long long)m[0]->sms * (ab ? PAIR_AB_BLOCKS : PAIR_BLOCKS) * PAIR_WARPS;
    const int band = pair_band_rows(m, n, GENERAL ? slots - slots / 16 : slots, width);
    p.split = GENERAL ? pair_split(band) : 1;
    int tiles = 0;
    for (int q = 0; q < n; ++q) {
        const State& s = *m[q];
        p.a[q] = make_args<float>(s);
        p.out[q] = s.f2;
        p.info[q] = s.pinfo;
        p.special[q] = s.pspecial;
        p.tile_begin[q] = tiles;
        p.strips[q] = pair_strips(s.nx, width);
        p.inv_d[q] = 1.0f / (float)p.strips[q];
        p.band[q] = band;
        const long long warps = (long long)p.strips[q] * ((s.ny + band - 1) / band);
        tiles += p.split * (int)((warps + PAIR_WARPS - 1) / PAIR_WARPS);
    }
    p.tile_begin[n] = tiles;
    if constexpr (ab) return launch_chained(k_step_ab_pair<S, MAXL>, tiles, PAIR_WARPS * 32, st, p);
    else return launch_chained(k_step_pair<S, GENERAL, GMODE, MAXL>, tiles, PAIR_WARPS * 32, st, p);
}

template <typename S, bool GENERAL>
static cudaError_t launch_pair_g(const State* const* m, int n, cudaStream_t st) {
    if constexpr (!GENERAL) {
        if (m[0]->g_mode == G_CURRENT)
            return n <= 4 ? launch_pair<S, false, G_CURRENT, 4>(m, n, st)
                          : launch_pair<S, false, G_CURRENT, GROUP_MAX>(m, n, st);
    }
    if (m[0]->g_mode == G_OFF)
        return n <= 4 ? launch_pair<S, GENERAL, G_OFF, 4>(m, n, st) : launch_pair<S, GENERAL, G_OFF, GROUP_MAX>(m, n, st);
    return n <= 4 ? launch_pair<S, GENERAL, G_LAGGED, 4>(m, n, st)
                  : launch_pair<S, GENERAL, G_LAGGED, GROUP_MAX>(m, n, st);
}

template <typename S>
cudaError_t Ops<S>::pair_maps(const State& s, unsigned* info, unsigned* special, cudaStream_t st) {
    if constexpr (sizeof(S) <= 4) {
        const Args<float> a = make_args<float>(s);
        const int strips = pair_strips(s.nx), words = (s.ny + 31) / 32;
        const cudaError_t e = cudaMemsetAsync(special, 0, sizeof(unsigned) * (size_t)strips * words, st);
        if (e != cudaSuccess) return e;
        const dim3 b(32, 8);
        k_pair_info<<<grid2d(s, b), b, 0, st>>>(a, info);
        const long long warps = (long long)strips * s.ny;
        k_pair_special<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(a, info, special, strips, words);
        return cudaGetLastError();
    } else {
        (void)s; (void)info; (void)special; (void)st;
        return cudaErrorInvalidValue;
    }
}

template <typename S>
cudaError_t Ops<S>::step_pair(const State* const* m, int n, cudaStream_t st) {
    if constexpr (sizeof(S) <= 4) {
        for (int q = 0; q < n; ++q)
            if (!m[q]->f2) return cudaErrorInvalidValue;
        for (int q0 = 0; q0 < n; q0 += GROUP_MAX) {
            const int c = n - q0 < GROUP_MAX ? n - q0 : GROUP_MAX;
            const cudaError_t e = m[q0]->general ? launch_pair_g<S, true>(m + q0, c, st)
                                                 : launch_pair_g<S, false>(m + q0, c, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    } else {
        (void)m; (void)n; (void)st;
        return cudaErrorInvalidValue;
    }
}

template <typename S>
cudaError_t Ops<S>::ghost_pass(const State& s, cudaStream_t st) {
    if (s.nghost <= 0) return cudaSuccess;
    using C = typename Fmt<S>::C;
    const Args<C> a = make_args<C>(s);
    const int t = 128, g = (s.nghost + t - 1) / t;
    if (s.parity == 0) launch_chained(k_ghosts<S, true>, g, t, st, a, s.ghosts, s.nghost);
    else launch_chained(k_ghosts<S, false>, g, t, st, a, s.ghosts, s.nghost);
    return cudaGetLastError();
}

}  // namespace trt
