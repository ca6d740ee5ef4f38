// Two time steps in one launch, for lattices periodic in x and y without a mask
// (lagged Phi or no G; FP32 and 16-bit storage).
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
// The same arithmetic in the same order as two single steps, each population
// rounded to the storage type between them: the same bits.
//
// Measured on GB300, one lattice, us per step, single steps (vector kernel) /
// this kernel: FP32 4096^2 227.4 / 126.0 (133 GLUPS; the 44 B per node of a step
// are 111 us at the copy bandwidth), 2048^2 62.7 / 33.4, 1024^2 15.4 / 10.2,
// 512^2 7.3 / 5.2, 250 x 246 4.1 / 3.1; FP16 4096^2 147.0 / 105.2, 2048^2 42.1 /
// 29.2, 1024^2 12.8 / 9.8, 512^2 6.2 / 4.7.  FP32 at 4096^2 is near its traffic;
// the rest is bound by issue (FP16 77 % of the slots, 187 instructions per node
// and step) and, below 1024^2, by the walk of the band.  4 resident CTAs of 4
// warps (128 registers, no spills); 5 for the 16-bit formats (102 registers)
// were slower (4096^2 108.8, 1024^2 11.3).
#pragma once
#include "lb_batch.cuh"
#include "lb_device.cuh"
#include "lb_vec.cuh"

namespace trt {

constexpr int PAIR_ROWS = 128, PAIR_ROWS_MIN = 2;   // rows of a band
inline int pair_strips(int nx) { return (nx + PAIR_W - 1) / PAIR_W; }

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
constexpr int PAIR_BLOCKS = 4;

// Rows per band for n lattices sharing a launch: the smallest number with which
// every warp is resident at once, or, where that is more than PAIR_ROWS, in the
// fewest whole waves of bands of at most PAIR_ROWS rows.  A band's walk is
// sequential, so a partial wave costs a whole one: 4096^2 FP32 with 1.25, 1.5
// and 2 waves of shorter bands 157, 149 and 128 us per step against 126.0 in
// one; 250 x 246 with bands of 16, 8, 4 and 2 rows 7.15, 5.12, 4.11 and 3.09.
inline int pair_band_rows(const State* const* m, int n, long long slots) {
    auto warps = [&](int h) {
        long long w = 0;
        for (int q = 0; q < n; ++q) {
            const long long k = (long long)pair_strips(m[q]->nx) * ((m[q]->ny + h - 1) / h);
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

template <int MAXL> struct PairParams {
    int n;                       // lattices in this launch
    int tile_begin[MAXL + 1];    // prefix sums of CTAs
    int strips[MAXL];            // column strips of PAIR_W nodes
    int band[MAXL];              // rows per band
    float inv_d[MAXL];           // 1 / strips, rounded
    void* out[MAXL];             // the other population buffer
    Args<float> a[MAXL];
};

template <typename S, int GMODE, int MAXL>
__global__ void __launch_bounds__(PAIR_WARPS * 32, PAIR_BLOCKS)
    k_step_pair(const __grid_constant__ PairParams<MAXL> p) {
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
    const int nx = a.nx, ny = a.ny, pitch = a.pitch;
    const int strips = p.strips[lo], band_h = p.band[lo];
    const int lane = (int)threadIdx.x & 31;
    const int w = (b - p.tile_begin[lo]) * PAIR_WARPS + ((int)threadIdx.x >> 5);
    int band, strip;
    tile_divmod(w, strips, p.inv_d[lo], band, strip);
    const int y0 = band * band_h;
    if (y0 >= ny) return;   // the whole warp leaves together
    const int y1 = y0 + band_h < ny ? y0 + band_h : ny;

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
    S* __restrict__ O = static_cast<S*>(p.out[lo]);
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
        {
            float d[9], e[9], oa[9], ob[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                d[i] = K::lo(D[i]);
                e[i] = K::hi(D[i]);
            }
            collide<float>(d, dpx.x, dpy.x, a.k1, a.k1lo, a.k2, a.k2lo, a.kf, a.gx, a.gy, a.hgx, a.hgy, a.rho0, oa,
                           hx.x, hy.x);
            collide<float>(e, dpx.y, dpy.y, a.k1, a.k1lo, a.k2, a.k2lo, a.kf, a.gx, a.gy, a.hgx, a.hgy, a.rho0, ob,
                           hx.y, hy.y);
#pragma unroll
            for (int i = 0; i < 9; ++i) N[i] = K::make(oa[i], ob[i]);
        }
        // second step at row q = r - 1, from rows q - 1, q and r
        if (r > y0) {
            float d[9], e[9], oa[9], ob[9];
            const P E[9] = {C0, K::up(C1), B2, K::down(C3), N[4], K::up(B5), K::down(B6), K::down(N[7]), K::up(N[8])};
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                d[i] = K::lo(E[i]);
                e[i] = K::hi(E[i]);
            }
            float2 qx = make_float2(0.f, 0.f), qy = make_float2(0.f, 0.f), kx, ky;
            if (GMODE == G_LAGGED) {
                const float l = shfl_up1(hxc.y), rr = shfl_down1(hxc.x);
                qx = make_float2(0.5f * (hxc.y - l), 0.5f * (rr - hxc.x));
                qy = make_float2(0.5f * (hy.x - hym.x), 0.5f * (hy.y - hym.y));
            }
            collide<float>(d, qx.x, qy.x, a.k1, a.k1lo, a.k2, a.k2lo, a.kf, a.gx, a.gy, a.hgx, a.hgy, a.rho0, oa,
                           kx.x, ky.x);
            collide<float>(e, qx.y, qy.y, a.k1, a.k1lo, a.k2, a.k2lo, a.kf, a.gx, a.gy, a.hgx, a.hgy, a.rho0, ob,
                           kx.y, ky.y);
            const unsigned at = oq + (unsigned)c;
            if (st_b) {
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    *reinterpret_cast<P*>(O + opp(i) * plane + at) = K::make(oa[i], ob[i]);
                if (GMODE == G_LAGGED) {
                    *reinterpret_cast<float2*>(a.phi_out + at) = kx;
                    *reinterpret_cast<float2*>(a.phi_out + plane + at) = ky;
                }
            } else if (st_a) {
#pragma unroll
                for (int i = 0; i < 9; ++i) O[opp(i) * plane + at] = Fmt<S>::st(oa[i]);
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

}  // namespace trt
