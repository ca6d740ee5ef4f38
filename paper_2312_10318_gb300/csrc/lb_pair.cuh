// Two time steps in one launch (lagged Phi or no G; FP32 and 16-bit storage).
//
// A step on its own is bound by HBM (FP32, 88 B per node) or by its launch and
// tail (lattices in L2); two steps together read and write the state once.  The
// kernel goes from an odd level to the next one: there the post-collision
// population f*_i of a node sits in the node's own slot, plane ibar, so the
// first step pulls f_i from x - e_i, and what the second step stores is aligned.
// It reads one population buffer and writes the other (a node's neighbours
// read its old state whenever they get there), and one Phi buffer each.
//
// A warp owns a strip of 64 columns and a band of rows, two columns per lane,
// and walks down the band.  Per row it loads the nine populations of its columns
// once (from the rows r - 1, r and r + 1 they stream from), takes the x-shifted
// ones from the neighbouring lanes, collides row r (first step) and then row
// r - 1 (second step), whose nine populations come from the three rows of first-
// step results that the walk keeps in registers.  Nothing goes through shared
// memory and no warp waits for another.  Each step makes one column on either
// side of the strip stale: of the 64, 60 (lanes 1 to 30) are stored, and two
// rows per band are collided once more than they are stored.  The next row's
// loads are issued before the two collisions that hide them.
//
// On a lattice with walls, a mask or open edges, tiles (a strip's band) whose
// nodes and links are all plain take the same walk (pair_walk); the others
// pair_walk_general, which looks at one word per node.
//
// The same arithmetic in the same order as two single steps, each population
// rounded to the storage type between them: the same bits.  Which runs take it:
// lb_pair_rule.h.
//
// Measured on GB300, us per step, single steps / this kernel: FP32 4096^2 227 /
// 123, 1024^2 15.4 / 8.1; FP16 2048^2 42.1 / 27.4; whole solves, ms: creeping flow
// 4096 x 2048 FP32, 50 steps, 7.5 / 4.3, channel 2048 x 1024 FP16, 200 steps, 4.9 /
// 3.3.  FP32 at 4096^2 is near its traffic (44 B per node and step, 111 us at the
// copy bandwidth); the rest waits for its own results at 16 warps per SM (4
// resident CTAs of 4 warps, 125 of 128 registers, no spills).  The two collisions
// of a lane run in packed FP32 (f2), half the issue slots of two scalar ones.
#pragma once
#include "lb_batch.cuh"
#include "lb_device.cuh"
#include "lb_vec.cuh"

namespace trt {

constexpr int PAIR_ROWS = 128, PAIR_ROWS_MIN = 2;   // rows of a band

// ---- two consecutive nodes of one population ----------------------------------
// up(p): [x - 1, x] of the pair at [x, x + 1]; down(p): [x + 1, x + 2].
template <typename S> struct Pr;
template <> struct Pr<float> {
    using P = float2;
    static __device__ __forceinline__ P make(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ P join(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ float first(const P& p) { return p.x; }
    static __device__ __forceinline__ float second(const P& p) { return p.y; }
    static __device__ __forceinline__ float lo(const P& p) { return p.x; }
    static __device__ __forceinline__ float hi(const P& p) { return p.y; }
    static __device__ __forceinline__ P up(const P& p) { return make_float2(shfl_up1(p.y), p.x); }
    static __device__ __forceinline__ P down(const P& p) { return make_float2(p.y, shfl_down1(p.x)); }
};
template <typename H> struct Pr16 {
    using P = unsigned int;
    static __device__ __forceinline__ P make(float a, float b) { return Cvt2<H>::from_floats(a, b); }
    static __device__ __forceinline__ P join(H a, H b) {
        return (unsigned)*reinterpret_cast<const unsigned short*>(&a) |
               ((unsigned)*reinterpret_cast<const unsigned short*>(&b) << 16);
    }
    static __device__ __forceinline__ H half_of(unsigned short b) { return *reinterpret_cast<const H*>(&b); }
    static __device__ __forceinline__ H first(const P& p) { return half_of((unsigned short)(p & 0xffffu)); }
    static __device__ __forceinline__ H second(const P& p) { return half_of((unsigned short)(p >> 16)); }
    static __device__ __forceinline__ float lo(const P& p) { return Cvt2<H>::to_float2(p).x; }
    static __device__ __forceinline__ float hi(const P& p) { return Cvt2<H>::to_float2(p).y; }
    static __device__ __forceinline__ P up(const P& p) { return __byte_perm(shfl_up1(p), p, 0x5432); }
    static __device__ __forceinline__ P down(const P& p) { return __byte_perm(p, shfl_down1(p), 0x5432); }
};
template <> struct Pr<__half> : Pr16<__half> {};
template <> struct Pr<__nv_bfloat16> : Pr16<__nv_bfloat16> {};

// Resident CTAs per SM the two-step kernel asks the compiler to allow.
constexpr int PAIR_BLOCKS = 4, PAIR_AB_BLOCKS = 3, PAIR_AB_AHEAD = 3;

// Rows per band for n lattices sharing a launch: the smallest number with which
// every warp is resident at once, or, where that is more than PAIR_ROWS, in the
// fewest whole waves of bands of at most PAIR_ROWS rows.  A band's walk is
// sequential, so a partial wave costs a whole one: 4096^2 FP32 in one wave 126 us
// per step, in 1.25 waves of shorter bands 157; and a small lattice's launch is as
// long as one walk: 250 x 246 with bands of 16 and 2 rows 7.2 and 3.1.
inline int pair_band_rows(const State* const* m, int n, long long slots, int width) {
    auto warps = [&](int h) {
        long long w = 0;
        for (int q = 0; q < n; ++q) {
            const long long k = (long long)pair_strips(m[q]->nx, width) * ((m[q]->ny + h - 1) / h);
            w += (k + PAIR_WARPS - 1) / PAIR_WARPS * PAIR_WARPS;
        }
        return w;
    };
    const long long fit = (warps(PAIR_ROWS) + slots - 1) / slots * slots;
    int lo = PAIR_ROWS_MIN, hi = PAIR_ROWS;
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (warps(mid) <= fit) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// Parts of a tile of a general lattice that is not plain.  Its rows take longer
// (walls on the way in and out, elementwise loads), and in one wave the longest
// walk is the launch's length: such a tile is walked by up to 8 warps of at least
// 8 rows each.  They come first; where the tile is plain they leave at once.
// Whole solves, ms, unsplit / split: creeping flow 4096 x 2048 FP32 6.2 / 4.4,
// channel 2048 x 1024 FP16 (bands of 16 rows) 4.2 / 3.5.
inline int pair_split(int band) { return band < 16 ? 1 : (band >= 64 ? 8 : band / 8); }

template <int MAXL> struct PairParams {
    int n;                       // lattices in this launch
    int split;                   // parts of a tile that is not plain (general lattices)
    int tile_begin[MAXL + 1];    // prefix sums of CTAs
    int strips[MAXL];            // column strips of PAIR_W nodes
    int band[MAXL];              // rows per band
    float inv_d[MAXL];           // 1 / strips, rounded
    void* out[MAXL];             // the other population buffer
    const unsigned* info[MAXL];     // general lattices: State::pinfo, State::pspecial
    const unsigned* special[MAXL];
    Args<float> a[MAXL];
};

// The collision of a pair's two nodes, packed; results rounded to storage.
template <typename S>
__device__ __forceinline__ void collide_pair(const Args<float>& a, const typename Pr<S>::P (&D)[9], float2 dpx, float2 dpy,
                                             typename Pr<S>::P (&N)[9], float2& hx, float2& hy) {
    using K = Pr<S>;
    f2 d[9], o[9], px, py;
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = f2(K::lo(D[i]), K::hi(D[i]));
    auto both = [](float v) { return f2(v, v); };
    collide_from<f2>(node_moments<f2>(d, both(a.hgx), both(a.hgy), both(a.rho0)), f2(dpx.x, dpx.y), f2(dpy.x, dpy.y),
                     both(a.k1), both(a.k1lo), both(a.k2), both(a.k2lo), both(a.kf), both(a.gx), both(a.gy), o, px, py);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        float u, v;
        unpk(o[i].v, u, v);
        N[i] = K::make(u, v);
    }
    unpk(px.v, hx.x, hx.y);
    unpk(py.v, hy.x, hy.y);
}

// The walk of one warp down rows y0 .. y1 - 1 of a strip whose rows y0 - 1 .. y1
// hold plain fluid nodes only, none of them linked to anything else.
template <typename S, int GMODE>
__device__ __forceinline__ void pair_walk(const Args<float>& a, S* __restrict__ O, int strip, int y0, int y1, int lane) {
    using K = Pr<S>;
    using P = typename K::P;
    const int nx = a.nx, ny = a.ny, pitch = a.pitch;

    // this lane's two columns c, c + 1 and where they lie in the lattice
    const int c = strip * PAIR_W - 2 + 2 * lane;
    int ca = c < 0 ? c + nx : c, cb = c + 1 < 0 ? c + 1 + nx : c + 1;
    if (ca >= nx) ca %= nx;
    if (cb >= nx) cb %= nx;
    const bool pair_ok = !(ca & 1) && cb == ca + 1;
    const bool vec = __all_sync(0xffffffffu, pair_ok);
    const bool inner = lane >= 1 && lane <= 30;
    const bool st_a = inner && c < nx, st_b = inner && c + 1 < nx;

    const S* __restrict__ F = static_cast<const S*>(a.f);
    const long long plane = a.plane;

    // the row that is loaded next, and the offsets of it and its two neighbours
    int yl = y0 == 0 ? ny - 1 : y0 - 1;
    unsigned om = (unsigned)((yl == 0 ? ny - 1 : yl - 1) * pitch), oc = (unsigned)(yl * pitch);
    int yn = yl == ny - 1 ? 0 : yl + 1;
    unsigned op = (unsigned)(yn * pitch);

    P L[9];
    float2 lpx = make_float2(0.f, 0.f), lpy = make_float2(0.f, 0.f);   // Phi_xxx of the row, Phi_yyy of the next
    auto load_row = [&]() {
        if (vec) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const unsigned r = (ey(i) > 0 ? om : (ey(i) < 0 ? op : oc)) + (unsigned)ca;
                L[i] = *reinterpret_cast<const P*>(F + opp(i) * plane + r);
            }
            if (GMODE == G_LAGGED) {
                lpx = *reinterpret_cast<const float2*>(a.phi_in + (oc + (unsigned)ca));
                lpy = *reinterpret_cast<const float2*>(a.phi_in + plane + (op + (unsigned)ca));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const unsigned r = ey(i) > 0 ? om : (ey(i) < 0 ? op : oc);
                const S* q = F + opp(i) * plane + r;
                L[i] = K::join(q[ca], q[cb]);
            }
            if (GMODE == G_LAGGED) {
                lpx = make_float2(a.phi_in[oc + (unsigned)ca], a.phi_in[oc + (unsigned)cb]);
                const float* q = a.phi_in + plane + op;
                lpy = make_float2(q[ca], q[cb]);
            }
        }
        om = oc;
        oc = op;
        yn = yn == ny - 1 ? 0 : yn + 1;
        op = (unsigned)(yn * pitch);
    };

    // Phi_yyy of the previous level in the rows above and at the loaded one
    float2 pym = make_float2(0.f, 0.f), pyc = make_float2(0.f, 0.f);
    if (GMODE == G_LAGGED) {
        const float* q = a.phi_in + plane;
        pym = make_float2(q[om + (unsigned)ca], q[om + (unsigned)cb]);
        pyc = make_float2(q[oc + (unsigned)ca], q[oc + (unsigned)cb]);
    }
    load_row();

    P B2{}, B5{}, B6{};                            // row q - 1: the populations going up
    P C0{}, C1{}, C3{}, C2{}, C5{}, C6{};          // row q
    float2 hxc = make_float2(0.f, 0.f);            // Phi_xxx of row q at the level between
    float2 hym = make_float2(0.f, 0.f), hyc = make_float2(0.f, 0.f);   // Phi_yyy of rows q - 1, q
    unsigned oq = 0;                               // row q = the row stored
    for (int r = y0 - 1; r <= y1; ++r) {
        // first step at row r, from the populations loaded
        P D[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) D[i] = ex(i) == 0 ? L[i] : (ex(i) > 0 ? K::up(L[i]) : K::down(L[i]));
        float2 dpx = make_float2(0.f, 0.f), dpy = make_float2(0.f, 0.f);
        if (GMODE == G_LAGGED) {
            const float l = shfl_up1(lpx.y), rr = shfl_down1(lpx.x);
            dpx = make_float2(0.5f * (lpx.y - l), 0.5f * (rr - lpx.x));
            dpy = make_float2(0.5f * (lpy.x - pym.x), 0.5f * (lpy.y - pym.y));
            pym = pyc;
            pyc = lpy;
        }
        if (r < y1) load_row();                    // the next row's, while this one collides
        P N[9];
        float2 hx, hy;
        collide_pair<S>(a, D, dpx, dpy, N, hx, hy);
        // second step at row q = r - 1, from rows q - 1, q and r
        if (r > y0) {
            const P E[9] = {C0, K::up(C1), B2, K::down(C3), N[4], K::up(B5), K::down(B6), K::down(N[7]), K::up(N[8])};
            P M[9];
            float2 qx = make_float2(0.f, 0.f), qy = make_float2(0.f, 0.f), kx, ky;
            if (GMODE == G_LAGGED) {
                const float l = shfl_up1(hxc.y), rr = shfl_down1(hxc.x);
                qx = make_float2(0.5f * (hxc.y - l), 0.5f * (rr - hxc.x));
                qy = make_float2(0.5f * (hy.x - hym.x), 0.5f * (hy.y - hym.y));
            }
            collide_pair<S>(a, E, qx, qy, M, kx, ky);
            const unsigned at = oq + (unsigned)c;
            if (st_b) {
#pragma unroll
                for (int i = 0; i < 9; ++i) *reinterpret_cast<P*>(O + opp(i) * plane + at) = M[i];
                if (GMODE == G_LAGGED) {
                    *reinterpret_cast<float2*>(a.phi_out + at) = kx;
                    *reinterpret_cast<float2*>(a.phi_out + plane + at) = ky;
                }
            } else if (st_a) {
#pragma unroll
                for (int i = 0; i < 9; ++i) O[opp(i) * plane + at] = K::first(M[i]);
                if (GMODE == G_LAGGED) {
                    a.phi_out[at] = kx.x;
                    a.phi_out[plane + at] = ky.x;
                }
            }
        }
        oq = (unsigned)(r * pitch);   // r = y0 - 1 is never stored
        B2 = C2; B5 = C5; B6 = C6;
        C0 = N[0]; C1 = N[1]; C3 = N[3]; C2 = N[2]; C5 = N[5]; C6 = N[6];
        hxc = hx;
        hym = hyc;
        hyc = hy;
    }
}

// ---- walls, masks and open edges -----------------------------------------------
// What a node's two steps need of its surroundings, one word per node of a
// general lattice: bit i - 1: f_i arrives from a wall (x - e_i is solid, a moving
// wall or outside), so it is the node's own f*_ibar of the step before; bit
// 7 + i: f*_i leaves into a moving wall (Ladd's correction); bits 16 ..: class.
enum : unsigned { PI_CLASS_SHIFT = 16, PI_OUTSIDE = 0xffu | ((unsigned)SOLID << PI_CLASS_SHIFT) };

static __global__ void k_pair_info(Args<float> a, unsigned* info) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= a.nx || y >= a.ny) return;
    int nb[9], kind[9];
    links<true>(a, x, y, nb, kind);
    unsigned v = (unsigned)(a.mask ? a.mask[nb[0]] : FLUID) << PI_CLASS_SHIFT;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        if (kind[opp(i)] != K_STREAM) v |= 1u << (i - 1);
        if (kind[i] == K_MOVING) v |= 1u << (7 + i);
    }
    info[nb[0]] = v;
}

// Bit y % 32 of special[strip][y / 32]: a node of the strip's 64 columns in row y
// is not plain fluid or has a link that is not.  One warp per strip and row.
static __global__ void k_pair_special(Args<float> a, const unsigned* __restrict__ info, unsigned* special, int strips,
                                      int words) {
    const int lane = (int)threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * (blockDim.x / 32) + ((int)threadIdx.x >> 5);
    if (w >= (long long)strips * a.ny) return;   // the whole warp leaves together
    const int strip = (int)(w / a.ny), y = (int)(w % a.ny);
    bool any = false;
    for (int k = 0; k < 2; ++k) {
        const int c = strip * PAIR_W - 2 + 2 * lane + k;
        const bool in = (unsigned)c < (unsigned)a.nx;
        const int x = (c % a.nx + a.nx) % a.nx;
        any = any || (!in && !a.px) || info[(long long)y * a.pitch + x] != (unsigned)FLUID << PI_CLASS_SHIFT;
    }
    if (__any_sync(0xffffffffu, any) && lane == 0) atomicOr(&special[(long long)strip * words + (y >> 5)], 1u << (y & 31));
}

// The same walk over any nodes.  The first step reads each population of a node
// straight from the slot that holds it (an odd level's rule, pop_loc), so that it
// is valid on all 64 columns and the second on 62: an outlet ghost in the first
// column stored takes what its inward neighbour, one column before, emits.
template <typename S, int GMODE>
__device__ __forceinline__ void pair_walk_general(const Args<float>& a, S* __restrict__ O,
                                               const unsigned* __restrict__ info, int strip, int y0, int y1, int lane) {
    using K = Pr<S>;
    using P = typename K::P;
    const int nx = a.nx, ny = a.ny, pitch = a.pitch;
    const long long plane = a.plane;
    const S* __restrict__ F = static_cast<const S*>(a.f);
    const int c = strip * PAIR_W - 2 + 2 * lane;
    // columns c - 1 .. c + 2: wrapped, or, past an open edge, the nearest one (never
    // read as a neighbour there: those links are walls)
    int col[4];
    bool out[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int x = c - 1 + k;
        out[k] = !a.px && (unsigned)x >= (unsigned)nx;
        col[k] = a.px ? (x % nx + nx) % nx : (x < 0 ? 0 : (x >= nx ? nx - 1 : x));
    }
    const bool inner = lane >= 1 && lane <= 30;
    // rows: wrapped, or past an open edge the nearest one, and whether they lie there
    auto row_out = [&](int y) { return !a.py && (unsigned)y >= (unsigned)ny; };
    auto row_of = [&](int y) {
        return (unsigned)((a.py ? ((y % ny) + ny) % ny : (y < 0 ? 0 : (y >= ny ? ny - 1 : y))) * pitch);
    };
    auto load_info = [&](unsigned row, bool ro) {
        uint2 v;
        v.x = ro || out[1] ? (unsigned)PI_OUTSIDE : info[row + (unsigned)col[1]];
        v.y = ro || out[2] ? (unsigned)PI_OUTSIDE : info[row + (unsigned)col[2]];
        return v;
    };
    auto cls = [](unsigned v) { return (int)(v >> PI_CLASS_SHIFT); };
    auto phi_row = [&](int comp, unsigned row, bool o) {   // Phi of the level before at this lane's two nodes
        const float* q = a.phi_in + comp * plane + row;
        return make_float2(o || out[1] ? 0.f : q[col[1]], o || out[2] ? 0.f : q[col[2]]);
    };
    // one node's collision with its corrections into moving walls
    auto collide_node = [&](float (&d)[9], unsigned v, float dpx, float dpy, float (&o)[9], float& hx, float& hy) {
        if (cls(v) == PRESSURE) zh_fill<float>(d, a.zh_dr);
        collide<float>(d, dpx, dpy, a.k1, a.k1lo, a.k2, a.k2lo, a.kf, a.gx, a.gy, a.hgx, a.hgy, a.rho0, o, hx, hy);
        if (v & 0xff00u) {
#pragma unroll
            for (int i = 1; i < 9; ++i)
                if (v >> (7 + i) & 1u) o[i] -= a.corr[i];
        }
    };

    P C[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) C[i] = K::make(0.f, 0.f);
    P B2 = C[2], B5 = C[5], B6 = C[6];
    const float2 z2 = make_float2(0.f, 0.f);
    float2 hxc = z2, hym = z2, hyc = z2, pym = z2, pyc = z2;
    if (GMODE == G_LAGGED) {
        pym = phi_row(1, row_of(y0 - 2), row_out(y0 - 2));
        pyc = phi_row(1, row_of(y0 - 1), row_out(y0 - 1));
    }
    // the row loaded next, r, with r - 1 and r + 1; info is read a row ahead of that,
    // because it decides where the row's populations are
    unsigned rm = row_of(y0 - 2), r0 = row_of(y0 - 1), rp = row_of(y0);
    int yp = (int)(rp / (unsigned)pitch);
    uint2 vq = make_uint2(PI_OUTSIDE, PI_OUTSIDE), v = load_info(r0, row_out(y0 - 1)), vn = load_info(rp, row_out(y0));
    float l0 = 0.f, l3 = 0.f;          // Phi_xxx beside the strip (lanes 0 and 31)
    S la[9], lb[9];
    float2 lpx = z2, lpy = z2;
    // whether a row has a node that is not plain (all bits of a plain fluid node's
    // word are 0); the others skip what walls, ghosts and outlets need
    auto special = [](uint2 w) { return __any_sync(0xffffffffu, (w.x | w.y) != 0u) != 0; };
    auto load_row = [&](int r, uint2 w) {
        if (special(w)) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const unsigned row = ey(i) > 0 ? rm : (ey(i) < 0 ? rp : r0);
                const bool wa = i > 0 && (w.x >> (i > 0 ? i - 1 : 0) & 1u), wb = i > 0 && (w.y >> (i > 0 ? i - 1 : 0) & 1u);
                la[i] = F[(wa ? i : opp(i)) * plane + (wa ? r0 + (unsigned)col[1] : row + (unsigned)col[1 - ex(i)])];
                lb[i] = F[(wb ? i : opp(i)) * plane + (wb ? r0 + (unsigned)col[2] : row + (unsigned)col[2 - ex(i)])];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const S* q = F + opp(i) * plane + (ey(i) > 0 ? rm : (ey(i) < 0 ? rp : r0));
                la[i] = q[col[1 - ex(i)]];
                lb[i] = q[col[2 - ex(i)]];
            }
        }
        if (GMODE == G_LAGGED) {
            const bool ro = row_out(r);
            lpx = phi_row(0, r0, ro);
            lpy = phi_row(1, rp, row_out(r + 1));
            if (lane == 0) l0 = ro || out[0] ? 0.f : a.phi_in[r0 + (unsigned)col[0]];
            if (lane == 31) l3 = ro || out[3] ? 0.f : a.phi_in[r0 + (unsigned)col[3]];
        }
        rm = r0;
        r0 = rp;
        yp = yp == ny - 1 ? (a.py ? 0 : yp) : yp + 1;
        rp = (unsigned)(yp * pitch);
    };
    load_row(y0 - 1, v);
    bool above = true;                 // special(vq)
    for (int r = y0 - 1; r <= y1; ++r) {
        float d[9], e[9], oa[9], ob[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            d[i] = Fmt<S>::ld(la[i]);
            e[i] = Fmt<S>::ld(lb[i]);
        }
        const float2 px = lpx, own_y = pyc;
        float2 dpx = z2, dpy = z2;
        if (GMODE == G_LAGGED) {
            float l = shfl_up1(px.y), rr = shfl_down1(px.x);
            if (lane == 0) l = l0;
            if (lane == 31) rr = l3;
            dpx.x = 0.5f * ((cls(v.x) == PRESSURE ? px.x : px.y) - l);
            dpx.y = 0.5f * ((cls(v.y) == PRESSURE ? px.y : rr) - px.x);
            dpy = make_float2(0.5f * (lpy.x - pym.x), 0.5f * (lpy.y - pym.y));
            pym = pyc;
            pyc = lpy;
        }
        uint2 v2 = vn;
        if (r < y1) {
            v2 = load_info(rp, row_out(r + 2));
            load_row(r + 1, vn);
        }
        float2 hx, hy;
        collide_node(d, v.x, dpx.x, dpy.x, oa, hx.x, hy.x);
        collide_node(e, v.y, dpx.y, dpy.y, ob, hx.y, hy.y);
        P N[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) N[i] = K::make(oa[i], ob[i]);
        // outlet ghosts emit what their inward neighbour, one column before, does;
        // Phi of solid and moving-wall nodes does not change
        auto settle = [&](uint2 w, P (&n)[9], float2& gx, float2& gy, float2 keep_x, float2 keep_y) {
            const bool ga = cls(w.x) == OUTLET, gb = cls(w.y) == OUTLET;
            if (__any_sync(0xffffffffu, ga || gb)) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const P u = K::up(n[i]);
                    n[i] = K::join(ga ? K::first(u) : K::first(n[i]), gb ? K::second(u) : K::second(n[i]));
                }
                const float ux = shfl_up1(gx.y), uy = shfl_up1(gy.y);
                if (gb) gx.y = gx.x, gy.y = gy.x;
                if (ga) gx.x = ux, gy.x = uy;
            }
            if (!collides(cls(w.x)) && !ga) gx.x = keep_x.x, gy.x = keep_y.x;
            if (!collides(cls(w.y)) && !gb) gx.y = keep_x.y, gy.y = keep_y.y;
        };
        const bool here = special(v);
        if (here) settle(v, N, hx, hy, px, own_y);
        if (r > y0) {
            const P E[9] = {C[0], K::up(C[1]), B2, K::down(C[3]), N[4],
                            K::up(B5), K::down(B6), K::down(N[7]), K::up(N[8])};
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                d[i] = K::lo(E[i]);
                e[i] = K::hi(E[i]);
            }
            if (above) {
#pragma unroll
                for (int i = 1; i < 9; ++i) {
                    if (vq.x >> (i - 1) & 1u) d[i] = K::lo(C[opp(i)]);
                    if (vq.y >> (i - 1) & 1u) e[i] = K::hi(C[opp(i)]);
                }
            }
            float2 qx = z2, qy = z2, kx, ky;
            if (GMODE == G_LAGGED) {
                const float l = shfl_up1(hxc.y), rr = shfl_down1(hxc.x);
                qx.x = 0.5f * ((cls(vq.x) == PRESSURE ? hxc.x : hxc.y) - l);
                qx.y = 0.5f * ((cls(vq.y) == PRESSURE ? hxc.y : rr) - hxc.x);
                qy = make_float2(0.5f * (hy.x - hym.x), 0.5f * (hy.y - hym.y));
            }
            collide_node(d, vq.x, qx.x, qy.x, oa, kx.x, ky.x);
            collide_node(e, vq.y, qx.y, qy.y, ob, kx.y, ky.y);
            P M[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) M[i] = K::make(oa[i], ob[i]);
            if (above) settle(vq, M, kx, ky, kx, ky);
            const unsigned at = (unsigned)((r - 1) * pitch + c);
            const bool sa = inner && c < nx && (collides(cls(vq.x)) || cls(vq.x) == OUTLET);
            const bool sb = inner && c + 1 < nx && (collides(cls(vq.y)) || cls(vq.y) == OUTLET);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                S* q = O + opp(i) * plane + at;
                if (sa && sb) {
                    *reinterpret_cast<P*>(q) = M[i];
                } else {
                    if (sa) q[0] = K::first(M[i]);
                    if (sb) q[1] = K::second(M[i]);
                }
            }
            if (GMODE == G_LAGGED) {
                if (sa) a.phi_out[at] = kx.x, a.phi_out[plane + at] = ky.x;
                if (sb) a.phi_out[at + 1] = kx.y, a.phi_out[plane + at + 1] = ky.y;
            }
        }
        B2 = C[2]; B5 = C[5]; B6 = C[6];
#pragma unroll
        for (int i = 0; i < 9; ++i) C[i] = N[i];
        hxc = hx;
        hym = hyc;
        hyc = hy;
        vq = v;
        above = here;
        v = vn;
        vn = v2;
    }
}

template <typename S, bool GENERAL, int GMODE, int MAXL>
__global__ void __launch_bounds__(PAIR_WARPS * 32, PAIR_BLOCKS)
    k_step_pair(const __grid_constant__ PairParams<MAXL> p) {
    chain_begin();
    const int b = (int)blockIdx.x;
    int lo = 0, hi = p.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tile_begin[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    const Args<float>& a = p.a[lo];
    const int lane = (int)threadIdx.x & 31;
    int t = b - p.tile_begin[lo];
    int part = 0;                 // of a split tile
    if (GENERAL && p.split > 1) {
        const int one = (p.tile_begin[lo + 1] - p.tile_begin[lo]) / p.split;
        part = p.split - 1 - t / one;
        t -= (p.split - 1 - part) * one;
    }
    const int w = t * PAIR_WARPS + ((int)threadIdx.x >> 5);
    int band, strip;
    tile_divmod(w, p.strips[lo], p.inv_d[lo], band, strip);
    int y0 = band * p.band[lo];
    if (y0 >= a.ny) return;   // the whole warp leaves together
    int y1 = y0 + p.band[lo] < a.ny ? y0 + p.band[lo] : a.ny;
    S* O = static_cast<S*>(p.out[lo]);
    if (GENERAL) {
        // rows y0 - 1 .. y1, wrapped: row 0's and row ny - 1's walls make a band at
        // an open edge special, so the rows beyond it need no look
        bool any = false;
        const unsigned* sp = p.special[lo] + (long long)strip * ((a.ny + 31) / 32);
        for (int y = y0 - 1 + lane; y <= y1; y += 32) {
            const int yw = y < 0 ? a.ny - 1 : (y >= a.ny ? 0 : y);
            any = any || (sp[yw >> 5] >> (yw & 31) & 1u);
        }
        if (__any_sync(0xffffffffu, any)) {
            const int rows = (y1 - y0 + p.split - 1) / p.split;
            y0 += part * rows;
            y1 = y0 + rows < y1 ? y0 + rows : y1;
            if (y0 < y1) pair_walk_general<S, GMODE>(a, O, p.info[lo], strip, y0, y1, lane);
            return;
        }
        if (part > 0) return;
    }
    pair_walk<S, GMODE>(a, O, strip, y0, y1, lane);
}

// BYTES (4 or 8) from global to shared memory, asynchronously.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* to, const void* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from),
                 "n"(BYTES)
                 : "memory");
}

// ---- Phi at the current level -----------------------------------------------------
// Two time steps of the two-buffer step (lb_ab.cuh) on a lattice periodic in x and
// y without a mask, from the canonical f(t) in one buffer to f(t + 2) in the other.
// The same walk with Phi in it: loading row r gives its moments and Phi(t); row
// r - 1 collides (d_y Phi from rows r and r - 2, d_x from the lanes beside), which
// completes f(t + 1) of row r - 2, its moments and Phi(t + 1); row r - 3 collides,
// which completes f(t + 2) of row r - 4, stored aligned.  Moments are kept for the
// collision two rows later, the three rows of collided populations per step in
// registers.  Phi takes two columns more of either side than lagged Phi does: 56
// of 64 are stored, and a band of h rows loads h + 8.
//
// A step of its own moves 72 B per node (FP32) and the TMA-fed kernel issues 378
// instructions for it; two in one launch move 36 per step.  us per step, the
// kernels of single steps (TMA-fed, column, plain: the fastest) / this one: FP32
// 4096^2 229 / 128, 2048^2 61.3 / 34.9, 1024^2 16.0 / 12.7, 512^2 8.2 / 7.0; FP16
// 4096^2 178 / 120, 2048^2 53.0 / 33.5, 1024^2 16.4 / 12.2.  Bound by latency at 12
// warps per SM (168 registers; 4 CTAs spill: 2048^2 FP32 144).
template <typename S, int MAXL>
__global__ void __launch_bounds__(PAIR_WARPS * 32, PAIR_AB_BLOCKS)
    k_step_ab_pair(const __grid_constant__ PairParams<MAXL> p) {
    using K = Pr<S>;
    using P = typename K::P;
    chain_begin();
    const int b = (int)blockIdx.x;
    int lo = 0, hi = p.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tile_begin[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    const Args<float>& a = p.a[lo];
    const int lane = (int)threadIdx.x & 31;
    const int w = (b - p.tile_begin[lo]) * PAIR_WARPS + ((int)threadIdx.x >> 5);
    int band, strip;
    tile_divmod(w, p.strips[lo], p.inv_d[lo], band, strip);
    const int y0 = band * p.band[lo];
    const int nx = a.nx, ny = a.ny, pitch = a.pitch;
    if (y0 >= ny) return;   // the whole warp leaves together
    const int y1 = y0 + p.band[lo] < ny ? y0 + p.band[lo] : ny;
    const S* __restrict__ F = static_cast<const S*>(a.f);
    S* __restrict__ O = static_cast<S*>(p.out[lo]);
    const long long plane = a.plane;

    const int c = strip * PAIR_AB_W - 4 + 2 * lane;
    const int ca = ((c % nx) + nx) % nx, cb = ca + 1 == nx ? 0 : ca + 1;
    const bool vec = __all_sync(0xffffffffu, !(ca & 1) && cb == ca + 1);
    const bool inner = lane >= 2 && lane <= 29;
    const bool st_a = inner && c < nx, st_b = inner && c + 1 < nx;

    // FP32 rows arrive through a ring of shared memory that each lane fills for
    // itself (asynchronous copies, PAIR_AB_AHEAD - 1 rows in flight per warp): one
    // row ahead in registers kept 27 KB in flight per SM, a third of what HBM's
    // latency needs (2048^2 60 us per step, 35 with the ring).  16-bit rows, half
    // the bytes and four-byte copies, are loaded into registers one row ahead
    // (33.5, and 38.7 through the ring).
    constexpr bool RING = sizeof(S) == 4;
    __shared__ P ring[PAIR_WARPS][RING ? PAIR_AB_AHEAD : 1][9][32];
    P(*slot)[9][32] = ring[threadIdx.x >> 5];
    P ahead[9];
    const int rl = y1 + 3;                           // last row the band needs
    int yl = ((y0 - 4) % ny + ny) % ny, rn = y0 - 4; // the row copied next, wrapped and not
    auto copy_row = [&]() {
        if (rn <= rl) {
            const unsigned r = (unsigned)(yl * pitch);
            P(*to)[32] = slot[RING ? (rn - y0 + 4) % PAIR_AB_AHEAD : 0];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const S* q = F + i * plane + r;
                if constexpr (!RING) {
                    ahead[i] = vec ? *reinterpret_cast<const P*>(q + ca) : K::join(q[ca], q[cb]);
                } else if (vec) {
                    copy_async<8>(&to[i][lane], q + ca);
                } else {
                    copy_async<4>(&to[i][lane], q + ca);
                    copy_async<4>(reinterpret_cast<char*>(&to[i][lane]) + 4, q + cb);
                }
            }
            yl = yl == ny - 1 ? 0 : yl + 1;
        }
        ++rn;
        if (RING) asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto both = [](float v) { return f2(v, v); };
    auto moments = [&](const P (&E)[9]) {
        f2 d[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) d[i] = f2(K::lo(E[i]), K::hi(E[i]));
        return node_moments<f2>(d, both(a.hgx), both(a.hgy), both(a.rho0));
    };
    // the collision of a row from its moments and the Phi around it
    auto collide_row = [&](const NodeMom<f2>& m, f2 hx, f2 up, f2 down, P (&N)[9]) {
        float x0, x1;
        unpk(hx.v, x0, x1);
        const float l = shfl_up1(x1), r = shfl_down1(x0);
        const f2 half = f2(0.5);
        const f2 dpx = rmul(half, rsub(f2(x1, r), f2(l, x0))), dpy = rmul(half, rsub(up, down));
        f2 o[9], px, py;
        collide_from<f2>(m, dpx, dpy, both(a.k1), both(a.k1lo), both(a.k2), both(a.k2lo), both(a.kf), both(a.gx),
                         both(a.gy), o, px, py);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float u, v;
            unpk(o[i].v, u, v);
            N[i] = K::make(u, v);
        }
    };
    // three rows of collided populations, of which the middle one's streamed state
    // is complete when the third arrives
    struct Ring {
        P B2, B5, B6, C0, C1, C3, C2, C5, C6;
        __device__ __forceinline__ void take(const P (&N)[9], P (&E)[9]) {
            E[0] = C0; E[1] = K::up(C1); E[2] = B2; E[3] = K::down(C3); E[4] = N[4];
            E[5] = K::up(B5); E[6] = K::down(B6); E[7] = K::down(N[7]); E[8] = K::up(N[8]);
            B2 = C2; B5 = C5; B6 = C6;
            C0 = N[0]; C1 = N[1]; C3 = N[3]; C2 = N[2]; C5 = N[5]; C6 = N[6];
        }
    };
    const f2 zero = f2(0.0);
    Ring R{}, Q{};
    NodeMom<f2> mp{}, mq{};
    f2 hxp = zero, hyp = zero, hypp = zero, hxq = zero, hyq = zero, hyqq = zero;
#pragma unroll
    for (int k = 0; k < (RING ? PAIR_AB_AHEAD - 1 : 1); ++k) copy_row();
    for (int r = y0 - 4; r <= rl; ++r) {
        if (RING) asm volatile("cp.async.wait_group %0;" ::"n"(PAIR_AB_AHEAD - 2) : "memory");
        P L[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) L[i] = RING ? slot[(r - y0 + 4) % PAIR_AB_AHEAD][i][lane] : ahead[i];
        copy_row();                                  // into the slot read a row ago
        const NodeMom<f2> m = moments(L);
        const f2 hy = phi_of(m.rho, m.uy);
        if (r > y0 - 3) {                            // rows up to y0 - 4 do not collide
            P N[9], E[9];
            collide_row(mp, hxp, hy, hypp, N);       // row r - 1
            R.take(N, E);                            // f(t + 1) of row r - 2
            const NodeMom<f2> m2 = moments(E);
            const f2 hy2 = phi_of(m2.rho, m2.uy);
            if (r > y0 + 1) {
                collide_row(mq, hxq, hy2, hyqq, N);  // row r - 3
                Q.take(N, E);                        // f(t + 2) of row r - 4
                if (r >= y0 + 4) {
                    const unsigned at = (unsigned)((r - 4) * pitch + c);
                    if (st_b) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) *reinterpret_cast<P*>(O + i * plane + at) = E[i];
                    } else if (st_a) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) O[i * plane + at] = K::first(E[i]);
                    }
                }
            }
            mq = m2;
            hxq = phi_of(m2.rho, m2.ux);
            hyqq = hyq;
            hyq = hy2;
        }
        mp = m;
        hxp = phi_of(m.rho, m.ux);
        hypp = hyp;
        hyp = hy;
    }
}

}  // namespace trt
