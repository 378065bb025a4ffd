// The annular problem (Section 2.3 and the FD discussion of Section 2.4): a square with a
// square hole, Dirichlet data on the hole, a Robin condition du/dn - i k u = q on the
// outer edge.
//
// Grid: [-side/2, side/2]^2 with N intervals per axis (N a power of two), h = side / N,
// node (i, j) at (-side/2 + i h, -side/2 + j h), stored at i (N + 1) + j.  Node types:
// HOLE (|x|, |y| <= hole: Dirichlet, value g), EDGE (i or j in {0, N}: the row is the
// outward normal derivative, the one-sided difference towards the inward neighbour,
// averaged over the two normals at a corner), PDE (5-point Delta_h).
//
// Outer iteration (FP64, Section 2.3 in residual form, sigma = alpha - k^2 >= 0):
//   r_N = b - B U_N,  A_sigma e_N = r_N,  U_{N+1} = U_N + e_N,
// B: PDE rows Delta_h + k^2, EDGE rows d/dn - i k;  A_sigma: PDE rows Delta_h - sigma,
// EDGE rows d/dn.  With exact inner solves the partial sums are those of the paper's
// v_n + i w_n (Neumann data -k w_{n-1}, +k v_{n-1} on the outer edge).
//
// Inner solve: multigrid V-cycles in the inner precision on rediscretised levels N, N/2,
// ..., 8 (node types by the same rule at each level; the coarsest solved exactly through a
// host-computed inverse).  Red-black Gauss-Seidel solves each row by its own equation;
// the residual is restricted by full weighting at PDE nodes and injected at EDGE nodes;
// bilinear prolongation.  A coarse level represents the hole only to its own spacing, and
// the coarse-grid correction is poor in the layer between the fine and the coarse hole
// edges: after each correction a band of a few nodes around the hole is relaxed several
// times, which restores the cycle's contraction (about 0.3 per V(2,2) cycle).
#include "../../include/helm.h"
#include "launch.h"
#include "pdl.cuh"
#include "fp_bits.cuh"
#include "fixed_win.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

namespace helm {
namespace {

constexpr int AN_NT = 256;
constexpr int AN_NC = 8;            // coarsest level (solved exactly)
constexpr int AN_BAND = 4;          // band half-width around the hole, in nodes of the level
constexpr int AN_BAND_SWEEPS = 4;
constexpr size_t AN_SMEM_MAX = 227 * 1024;
enum : unsigned char { AN_PDE = 0, AN_EDGE = 1, AN_HOLE = 2 };

template <typename R> struct CX;
template <> struct CX<float> { typedef float2 T; };
template <> struct CX<double> { typedef double2 T; };
template <> struct CX<long long> { typedef longlong2 T; };     // fixed-point windows

__host__ __device__ constexpr size_t an_a16(size_t b) { return (b + 15) & ~(size_t)15; }

int grid_for(long work) { return (int)std::min<long>((work + AN_NT - 1) / AN_NT, 152L * 16); }

// FP64 <-> inner precision; complex64's format changes run on the integer pipes
__device__ __forceinline__ double an_widen(float x) { return f2d_bits(x); }
__device__ __forceinline__ double an_widen(double x) { return x; }
__device__ __forceinline__ float an_narrow(double x, float) { return d2f_bits(x); }
__device__ __forceinline__ double an_narrow(double x, double) { return x; }

// ---------------------------------------------------------------------------
// A level's side of the cycle in one launch, on windows in shared memory
// ---------------------------------------------------------------------------
// Windows are held as two colour planes (node (lx, ly) of the window, whose colour is
// (gx + gy) & 1, at ly * W / 2 + (lx >> 1) of its colour's plane; W even): a half-sweep
// reads and writes contiguous words.  Their nodes are numbered row by row over all the
// CTA's threads, and row types follow from the indices (the hole is an index box), so no
// type array is read.  Half-sweep k updates the nodes that lie k + 1 inside the window, so
// that every updated node sees the values of a full-grid sweep.
// A tile is T x T fine nodes (T / 2 coarse ones a side in the descent): 32, or 16 on the
// levels that 32 would cut into fewer tiles than there are SMs (an_tile).
constexpr int AN_TT = 512;           // threads of a tile CTA

// index boxes of a level: the hole [lo, hi]^2 and the band ring [b0, b1]^2 around it
struct AnGeo {
    int n, lo, hi, b0, b1;
    __device__ bool hole(int i, int j) const { return i >= lo && i <= hi && j >= lo && j <= hi; }
    __device__ bool edge(int i, int j) const { return i == 0 || i == n || j == 0 || j == n; }
};

// q / d for 0 <= q < 65536, 1 <= d <= 4096 by m = ceil(2^32 / d)
__device__ __forceinline__ unsigned an_magic(int d) { return 0xffffffffu / (unsigned)d + 1u; }
__device__ __forceinline__ int an_div(int q, int d, unsigned m) { return d == 1 ? q : (int)__umulhi((unsigned)q, m); }

// a window: origin (y0, x0), even row length W, colour planes of the iterate and the rhs
template <typename R> struct AnWin {
    typedef typename CX<R>::T c2;
    int y0, x0, W;
    c2 *E0, *E1, *R0, *R1;
    __device__ int at(int i, int j) const { return (i - y0) * (W >> 1) + ((j - x0) >> 1); }
    __device__ c2* E(int color) const { return color ? E1 : E0; }
    __device__ c2* Rh(int color) const { return color ? R1 : R0; }
    __device__ c2 e(int i, int j) const { return E((i + j) & 1)[at(i, j)]; }
};

// mean of the inward neighbours of edge node (i, j), held in the plane Eo
template <typename R>
__device__ __forceinline__ typename CX<R>::T inward_mean_w(const AnWin<R>& w, const typename CX<R>::T* Eo, int i,
                                                           int j, int n)
{
    typename CX<R>::T s;
    s.x = 0;
    s.y = 0;
    int c = 0;
    if (i == 0) { const auto v = Eo[w.at(1, j)]; s.x += v.x; s.y += v.y; ++c; }
    if (i == n) { const auto v = Eo[w.at(n - 1, j)]; s.x += v.x; s.y += v.y; ++c; }
    if (j == 0) { const auto v = Eo[w.at(i, 1)]; s.x += v.x; s.y += v.y; ++c; }
    if (j == n) { const auto v = Eo[w.at(i, n - 1)]; s.x += v.x; s.y += v.y; ++c; }
    if (c == 2) { s.x *= 0.5f; s.y *= 0.5f; }
    return s;
}

// One red-black half-sweep over rows ya..yb, columns xa..xb (inside the grid): PDE rows
// e = (sum of neighbours - h^2 rhs) / (4 + sigma h^2), EDGE rows the mean of the inward
// neighbours plus h rhs, hole nodes left alone.  PURE: PDE nodes only.
template <typename R, bool PURE>
__device__ __forceinline__ void an_half_w(const AnWin<R>& w, const AnGeo& g, int ya, int yb, int xa, int xb, R h,
                                          R dinv, int color)
{
    typedef typename CX<R>::T c2;
    if (ya > yb || xa > xb) return;
    const int nx = (xb - xa + 2) >> 1, total = nx * (yb - ya + 1);
    const unsigned m = an_magic(nx);
    const R h2 = h * h;
    c2* __restrict__ Ec = w.E(color);
    const c2* __restrict__ Eo = w.E(color ^ 1);
    const c2* __restrict__ Rc = w.Rh(color);
    for (int q = threadIdx.x; q < total; q += blockDim.x) {
        const int r = an_div(q, nx, m);
        const int i = ya + r;
        const int j = xa + ((xa + i + color) & 1) + 2 * (q - r * nx);
        if (j > xb) continue;
        if (!PURE && g.hole(i, j)) continue;
        const int o = w.at(i, j);
        const c2 rr = Rc[o];
        c2 v;
        if (PURE || !g.edge(i, j)) {
            const c2 a = Eo[w.at(i - 1, j)], b = Eo[w.at(i + 1, j)], c = Eo[w.at(i, j - 1)], d = Eo[w.at(i, j + 1)];
            v.x = (((a.x + b.x) + (c.x + d.x)) - h2 * rr.x) * dinv;
            v.y = (((a.y + b.y) + (c.y + d.y)) - h2 * rr.y) * dinv;
        } else {
            const c2 s = inward_mean_w<R>(w, Eo, i, j, g.n);
            v.x = s.x + h * rr.x;
            v.y = s.y + h * rr.y;
        }
        Ec[o] = v;
    }
}

// does the box hold neither edge nor hole nodes?
__device__ __forceinline__ bool an_pure(const AnGeo& g, int ya, int yb, int xa, int xb)
{
    return ya >= 1 && yb < g.n && xa >= 1 && xb < g.n && (yb < g.lo || ya > g.hi || xb < g.lo || xa > g.hi);
}

template <typename R>
__device__ __forceinline__ void an_half_any(const AnWin<R>& w, const AnGeo& g, int ya, int yb, int xa, int xb, R h,
                                            R dinv, int color)
{
    if (an_pure(g, ya, yb, xa, xb)) an_half_w<R, true>(w, g, ya, yb, xa, xb, h, dinv, color);
    else an_half_w<R, false>(w, g, ya, yb, xa, xb, h, dinv, color);
}

// nu sweeps of a window of `rows` rows whose outermost `skip` nodes are already spent
template <typename R>
__device__ __forceinline__ void an_sweeps_w(const AnWin<R>& w, const AnGeo& g, int rows, int cols, int skip, R h,
                                            R dinv, int nu)
{
    for (int k = 0; k < 2 * nu; ++k) {
        const int s = skip + k + 1;
        an_half_any<R>(w, g, max(0, w.y0 + s), min(g.n, w.y0 + rows - 1 - s), max(0, w.x0 + s),
                       min(g.n, w.x0 + cols - 1 - s), h, dinv, k & 1);
        __syncthreads();
    }
}

// the band sweeps (PDE rows of the ring) on such a window; its 2 AN_BAND_SWEEPS outermost
// nodes are spent afterwards
template <typename R>
__device__ __forceinline__ void an_band_w(const AnWin<R>& w, const AnGeo& g, int rows, int cols, bool whole, R h,
                                          R dinv)
{
    for (int k = 0; k < 2 * AN_BAND_SWEEPS; ++k) {
        const int s = whole ? 0 : k + 1;
        an_half_w<R, false>(w, g, max(g.b0, w.y0 + s), min(g.b1, w.y0 + rows - 1 - s), max(g.b0, w.x0 + s),
                            min(g.b1, w.x0 + cols - 1 - s), h, dinv, k & 1);
        __syncthreads();
    }
}

// stage rows x cols nodes of e (or zeros) and rhs (asynchronous copies; the caller waits)
template <typename R>
__device__ __forceinline__ void an_stage(const AnWin<R>& w, int rows, int cols, const typename CX<R>::T* __restrict__ e,
                                         const typename CX<R>::T* __restrict__ rhs, int n, bool load_e)
{
    typedef typename CX<R>::T c2;
    const int S = n + 1;
    const unsigned m = an_magic(cols);
    c2 z;
    z.x = 0;
    z.y = 0;
    for (int q = threadIdx.x; q < rows * cols; q += blockDim.x) {
        const int ly = an_div(q, cols, m), lx = q - ly * cols;
        const int i = w.y0 + ly, j = w.x0 + lx;
        const bool in = i >= 0 && i <= n && j >= 0 && j <= n;
        const size_t gq = in ? (size_t)i * S + j : 0;
        const int c = (i + j) & 1, o = w.at(i, j);
        if (load_e) cp_async_elem<sizeof(c2)>(w.E(c) + o, e + gq, in);
        else w.E(c)[o] = z;
        cp_async_elem<sizeof(c2)>(w.Rh(c) + o, rhs + gq, in);
    }
}

// residual of the row at (i, j): zero on the hole, rhs itself where the iterate is zero
template <typename R>
__device__ __forceinline__ typename CX<R>::T an_resid_w(const AnWin<R>& w, const AnGeo& g, int i, int j, R h, R ih2,
                                                        R sig, bool zero)
{
    typedef typename CX<R>::T c2;
    const int color = (i + j) & 1, o = w.at(i, j);
    c2 r = w.Rh(color)[o];
    if (g.hole(i, j)) { r.x = 0; r.y = 0; return r; }
    if (zero) return r;
    const c2 c = w.E(color)[o];
    const c2* __restrict__ Eo = w.E(color ^ 1);
    if (!g.edge(i, j)) {
        const c2 p = Eo[w.at(i - 1, j)], q = Eo[w.at(i + 1, j)], s = Eo[w.at(i, j - 1)], t = Eo[w.at(i, j + 1)];
        const R sx = (p.x + q.x) + (s.x + t.x), sy = (p.y + q.y) + (s.y + t.y);
        r.x -= (sx - (R)4 * c.x) * ih2 - sig * c.x;
        r.y -= (sy - (R)4 * c.y) * ih2 - sig * c.y;
    } else {
        const c2 mm = inward_mean_w<R>(w, Eo, i, j, g.n);
        r.x -= (c.x - mm.x) / h;
        r.y -= (c.y - mm.y) / h;
    }
    return r;
}

// coarse node (I, J) of the restriction of the fine residual, res(i, j) at fine nodes: full
// weighting at PDE nodes, injection at EDGE nodes, zero on the hole
template <typename R, typename F>
__device__ __forceinline__ typename CX<R>::T an_restrict_node(const AnGeo& gc, int I, int J, F res)
{
    typedef typename CX<R>::T c2;
    c2 v;
    if (gc.hole(I, J)) {
        v.x = 0;
        v.y = 0;
    } else if (gc.edge(I, J)) {
        v = res(2 * I, 2 * J);
    } else {
        R ax = 0, ay = 0;
#pragma unroll
        for (int a = -1; a <= 1; ++a)
#pragma unroll
            for (int b = -1; b <= 1; ++b) {
                const R wgt = (R)((2 - (a < 0 ? -a : a)) * (2 - (b < 0 ? -b : b)));
                const c2 r = res(2 * I + a, 2 * J + b);
                ax += wgt * r.x;
                ay += wgt * r.y;
            }
        v.x = ax * (R)(1.0 / 16.0);
        v.y = ay * (R)(1.0 / 16.0);
    }
    return v;
}

// ---- FP64 windows in 64-bit fixed point (fixed_win.cuh) ----
// PDE rows hold h^2 rhs, EDGE rows h rhs: e = mean of the inward neighbours + h rhs there.
// A 256^2 solve with V(2,2), 53 steps: 6.10 -> 3.95 ms.  The cycle's error against extended
// precision, N = 128 .. 512, two holes, rough / smooth / edge data: lower than the FP64
// windows' in 33 of 36 norms, the others (l2, 512, rough) 1.16e-15 against 1.00e-15 at most
// (tests/test_gpu_cycle_annulus.py holds one cycle to twice FP64's own and ten roundings).
// sigma > 0, more sweeps, and windows out of the scale's range keep the FP64 code.  Three or four
// descent sweeps would fit on a scale one bit coarser, which raised that error in 4 of 36 norms
// (by up to 1.7): they stay in FP64.
constexpr int AN_FX_NU1 = 2, AN_FX_NU2 = 4;      // most sweeps of a window in fixed point

// this thread's staged words (an_stage's numbering) of the window: their largest exponent
__device__ __forceinline__ int an_fx_exp(const AnWin<double>& w, const AnGeo& g, int rows, int cols, bool load_e,
                                         const FxH2& fp, const FxH2& fe)
{
    const unsigned m = an_magic(cols);
    int ex = 0;
    for (int q = threadIdx.x; q < rows * cols; q += blockDim.x) {
        const int ly = an_div(q, cols, m), i = w.y0 + ly, j = w.x0 + (q - ly * cols);
        const int c = (i + j) & 1, o = w.at(i, j), er = fx_exp2(w.Rh(c)[o]);
        ex = max(ex, er ? er + (g.edge(i, j) ? fe.add : fp.add) : 0);
        if (load_e) ex = max(ex, fx_exp2(w.E(c)[o]));
    }
    return ex;
}

// ... and those words in place on the scale em
__device__ __forceinline__ AnWin<long long> an_fx_window(const AnWin<double>& w, const AnGeo& g, int rows, int cols,
                                                         bool load_e, const FxH2& fp, const FxH2& fe, int em)
{
    const AnWin<long long> f{w.y0, w.x0, w.W, reinterpret_cast<longlong2*>(w.E0), reinterpret_cast<longlong2*>(w.E1),
                             reinterpret_cast<longlong2*>(w.R0), reinterpret_cast<longlong2*>(w.R1)};
    const unsigned m = an_magic(cols);
    for (int q = threadIdx.x; q < rows * cols; q += blockDim.x) {
        const int ly = an_div(q, cols, m), i = w.y0 + ly, j = w.x0 + (q - ly * cols);
        const int c = (i + j) & 1, o = w.at(i, j);
        const double2 r = w.Rh(c)[o];
        f.Rh(c)[o] = g.edge(i, j) ? fe.q2(r, em) : fp.q2(r, em);
        if (load_e) f.E(c)[o] = fx_q2(w.E(c)[o], em);      // (zeros stay zero)
    }
    return f;
}

// mean of the inward neighbours of edge node (i, j), held in the plane Eo
__device__ __forceinline__ longlong2 an_fx_inward(const AnWin<long long>& w, const longlong2* Eo, int i, int j, int n)
{
    longlong2 s = make_longlong2(0, 0);
    int c = 0;
    auto add = [&](int a, int b) {
        const longlong2 v = Eo[w.at(a, b)];
        s.x += v.x;
        s.y += v.y;
        ++c;
    };
    if (i == 0) add(1, j);
    if (i == n) add(n - 1, j);
    if (j == 0) add(i, 1);
    if (j == n) add(i, n - 1);
    return c == 2 ? make_longlong2(fx_shr<1>(s.x), fx_shr<1>(s.y)) : s;
}

__device__ __forceinline__ void an_fx_half(const AnWin<long long>& w, const AnGeo& g, int ya, int yb, int xa, int xb,
                                           int color)
{
    if (ya > yb || xa > xb) return;
    const int nx = (xb - xa + 2) >> 1, total = nx * (yb - ya + 1);
    const unsigned m = an_magic(nx);
    const bool pure = an_pure(g, ya, yb, xa, xb);
    longlong2* __restrict__ Ec = w.E(color);
    const longlong2* __restrict__ Eo = w.E(color ^ 1);
    const longlong2* __restrict__ Rc = w.Rh(color);
    for (int q = threadIdx.x; q < total; q += blockDim.x) {
        const int r = an_div(q, nx, m), i = ya + r;
        const int j = xa + ((xa + i + color) & 1) + 2 * (q - r * nx);
        if (j > xb || (!pure && g.hole(i, j))) continue;
        const int o = w.at(i, j);
        if (pure || !g.edge(i, j)) {
            Ec[o] = fx_gs(Eo[w.at(i - 1, j)], Eo[w.at(i + 1, j)], Eo[w.at(i, j - 1)], Eo[w.at(i, j + 1)], Rc[o]);
        } else {
            const longlong2 s = an_fx_inward(w, Eo, i, j, g.n), rr = Rc[o];
            Ec[o] = make_longlong2(s.x + rr.x, s.y + rr.y);
        }
    }
}

__device__ __forceinline__ void an_fx_sweeps(const AnWin<long long>& w, const AnGeo& g, int rows, int cols, int skip,
                                             int nu)
{
    for (int k = 0; k < 2 * nu; ++k) {
        const int s = skip + k + 1;
        an_fx_half(w, g, max(0, w.y0 + s), min(g.n, w.y0 + rows - 1 - s), max(0, w.x0 + s),
                   min(g.n, w.x0 + cols - 1 - s), k & 1);
        __syncthreads();
    }
}

// h^2 (PDE) or h (EDGE) times the residual of the row at (i, j); zero on the hole
__device__ __forceinline__ longlong2 an_fx_resid(const AnWin<long long>& w, const AnGeo& g, int i, int j, bool zero)
{
    const int color = (i + j) & 1, o = w.at(i, j);
    longlong2 r = w.Rh(color)[o];
    if (g.hole(i, j)) return make_longlong2(0, 0);
    if (zero) return r;
    const longlong2 c = w.E(color)[o];
    const longlong2* __restrict__ Eo = w.E(color ^ 1);
    if (!g.edge(i, j)) {
        const longlong2 p = Eo[w.at(i - 1, j)], q = Eo[w.at(i + 1, j)], s = Eo[w.at(i, j - 1)], t = Eo[w.at(i, j + 1)];
        r.x -= ((p.x + q.x) + (s.x + t.x)) - 4 * c.x;
        r.y -= ((p.y + q.y) + (s.y + t.y)) - 4 * c.y;
    } else {
        const longlong2 mm = an_fx_inward(w, Eo, i, j, g.n);
        r.x -= c.x - mm.x;
        r.y -= c.y - mm.y;
    }
    return r;
}

__host__ __device__ constexpr int an_down_rows(int T, int nu1) { return T + 3 + 4 * nu1; }
__host__ __device__ constexpr int an_up_w(int T, int nu2, bool band)
{
    return T + 2 * (2 * nu2 + (band ? 2 * AN_BAND_SWEEPS : 0));
}
template <typename R> size_t an_down_bytes(int T, int nu1)
{
    return 2 * (size_t)an_down_rows(T, nu1) * (an_down_rows(T, nu1) + 1) * sizeof(typename CX<R>::T);
}
template <typename R> size_t an_up_bytes(int T, int nu2)
{
    const size_t W = an_up_w(T, nu2, true);
    return (2 * W * W + (W / 2 + 1) * (W / 2 + 1)) * sizeof(typename CX<R>::T);
}

template <typename R>
__device__ __forceinline__ AnWin<R> an_window(void* smem, int y0, int x0, int rows, int W)
{
    typedef typename CX<R>::T c2;
    const int pl = rows * (W >> 1);
    c2* b = reinterpret_cast<c2*>(smem);
    return AnWin<R>{y0, x0, W, b, b + pl, b + 2 * pl, b + 3 * pl};
}

// Descent of one level: nu1 sweeps, then the coarse rhs for the T / 2 x T / 2 coarse nodes from
// (I0, J0); the swept fine iterate goes to e_out on the T x T fine nodes from (2 I0, 2 J0): a
// separate buffer, since other CTAs stage their windows from e meanwhile.
// Bound by the latency of its phases (FP64: by an SM's FP64 rate).  complex64, cold: level
// 1024 34 -> 28.8 us, 512 16 -> 10.6, 128 12 -> 8.3 against rows by warps with type bytes and
// unbatched loads.
template <typename R, int T>
__global__ void __launch_bounds__(AN_TT, 2)
k_an_down(const typename CX<R>::T* __restrict__ e, typename CX<R>::T* __restrict__ e_out,
          const typename CX<R>::T* __restrict__ rhs, AnGeo g, R h, R dinv, R sig, R ih2, int nu1, int load_e,
          typename CX<R>::T* __restrict__ rc, AnGeo gc)
{
    typedef typename CX<R>::T c2;
    constexpr int AN_CT = T / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = g.n, nc = gc.n;
    const int ntc = (nc + AN_CT) / AN_CT;
    const int I0 = (blockIdx.x / ntc) * AN_CT, J0 = (blockIdx.x % ntc) * AN_CT;
    const int hw = 2 + 2 * nu1;               // low side; the high side needs 2 nu1
    const int rows = an_down_rows(T, nu1), W = rows + 1;
    const AnWin<R> w = an_window<R>(smem_raw, 2 * I0 - hw, 2 * J0 - hw, rows, W);
    pdl_wait();
    pdl_trigger();
    an_stage<R>(w, rows, rows, e, rhs, n, load_e != 0);
    cp_async_wait_all();
    const bool zero = nu1 == 0 && load_e == 0;
    const int Sc = nc + 1, S = n + 1;
    const int ci1 = min(nc, I0 + AN_CT - 1), cj1 = min(nc, J0 + AN_CT - 1);
    if constexpr (std::is_same<R, double>::value) {
        // Fixed point with room for the largest sum.  In units of the window's largest value a
        // sweep adds 5 / 4 at most (an EDGE row adds h rhs to a neighbour that h^2 rhs / 4 went
        // into): 7 / 2 after two sweeps, residuals below 29, rows of the full weighting below
        // 116 (2^56 * 116 < 2^63).
        __shared__ int sx[AN_TT / 32];
        const FxH2 fp(h * h), fe(h);
        const bool plain = nu1 <= AN_FX_NU1 && fx_bits(dinv) == fx_bits(0.25);
        const int em = block_max_exp<AN_TT>(plain ? an_fx_exp(w, g, rows, rows, load_e != 0, fp, fe) : 0, sx) + 2;
        if (plain && fp.usable(em) && fe.usable(em)) {
            const AnWin<long long> f = an_fx_window(w, g, rows, rows, load_e != 0, fp, fe, em);
            __syncthreads();
            an_fx_sweeps(f, g, rows, rows, 0, nu1);
            for (int q = threadIdx.x; q < 4 * AN_CT * AN_CT; q += AN_TT) {
                const int i = 2 * I0 + q / (2 * AN_CT), j = 2 * J0 + q % (2 * AN_CT);
                if (i <= n && j <= n) e_out[(size_t)i * S + j] = fx_d2(f.e(i, j), em);
            }
            const int ry0 = max(0, 2 * I0 - 1), ry1 = min(n, 2 * ci1 + 1);
            const int rx0 = max(0, 2 * J0 - 1), rx1 = min(n, 2 * cj1 + 1);
            const int nx = rx1 - rx0 + 1;
            const unsigned m = an_magic(nx);
            for (int q = threadIdx.x; q < nx * (ry1 - ry0 + 1); q += AN_TT) {
                const int r = an_div(q, nx, m), i = ry0 + r, j = rx0 + (q - r * nx);
                f.Rh((i + j) & 1)[f.at(i, j)] = an_fx_resid(f, g, i, j, zero);
            }
            __syncthreads();
            for (int q = threadIdx.x; q < AN_CT * AN_CT; q += AN_TT) {
                const int I = I0 + q / AN_CT, J = J0 + q % AN_CT;
                if (I > ci1 || J > cj1) continue;
                auto res = [&](int i, int j) -> longlong2 { return f.Rh((i + j) & 1)[f.at(i, j)]; };
                double2 v = make_double2(0.0, 0.0);
                if (gc.edge(I, J)) {
                    v = fe.over(res(2 * I, 2 * J), em);
                } else if (!gc.hole(I, J)) {
                    longlong2 t[3];
#pragma unroll
                    for (int a = -1; a <= 1; ++a) {
                        const longlong2 u = res(2 * I + a, 2 * J - 1), c = res(2 * I + a, 2 * J),
                                        d = res(2 * I + a, 2 * J + 1);
                        t[a + 1] = make_longlong2(fx_shr<2>((u.x + d.x) + 2 * c.x), fx_shr<2>((u.y + d.y) + 2 * c.y));
                    }
                    v = fp.over(make_longlong2((t[0].x + t[2].x) + 2 * t[1].x, (t[0].y + t[2].y) + 2 * t[1].y), em - 2);
                }
                rc[(size_t)I * Sc + J] = v;
            }
            return;
        }
    }
    __syncthreads();
    an_sweeps_w<R>(w, g, rows, rows, 0, h, dinv, nu1);
    {
        const int fi1 = min(n, 2 * I0 + 2 * AN_CT - 1), fj1 = min(n, 2 * J0 + 2 * AN_CT - 1);
        for (int q = threadIdx.x; q < 4 * AN_CT * AN_CT; q += AN_TT) {
            const int i = 2 * I0 + q / (2 * AN_CT), j = 2 * J0 + q % (2 * AN_CT);
            if (i <= fi1 && j <= fj1) e_out[(size_t)i * S + j] = w.e(i, j);
        }
    }
    // the fine residual once per node, in place of the window's rhs: rows / columns
    // 2 I0 - 1 .. 2 ci1 + 1 (within the grid)
    {
        const int ry0 = max(0, 2 * I0 - 1), ry1 = min(n, 2 * ci1 + 1);
        const int rx0 = max(0, 2 * J0 - 1), rx1 = min(n, 2 * cj1 + 1);
        const int nx = rx1 - rx0 + 1;
        const unsigned m = an_magic(nx);
        for (int q = threadIdx.x; q < nx * (ry1 - ry0 + 1); q += AN_TT) {
            const int r = an_div(q, nx, m), i = ry0 + r, j = rx0 + (q - r * nx);
            w.Rh((i + j) & 1)[w.at(i, j)] = an_resid_w<R>(w, g, i, j, h, ih2, sig, zero);
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < AN_CT * AN_CT; q += AN_TT) {
        const int I = I0 + q / AN_CT, J = J0 + q % AN_CT;
        if (I > ci1 || J > cj1) continue;
        rc[(size_t)I * Sc + J] = an_restrict_node<R>(
            gc, I, J, [&](int i, int j) -> c2 { return w.Rh((i + j) & 1)[w.at(i, j)]; });
    }
}

// e(i, j) += bilinear interpolation of the coarse iterate, ce(I, J)
template <typename R, typename F>
__device__ __forceinline__ typename CX<R>::T an_corrected(typename CX<R>::T v, int i, int j, F ce)
{
    const int I0 = i >> 1, I1 = (i + 1) >> 1, J0 = j >> 1, J1 = (j + 1) >> 1;
    const auto a = ce(I0, J0), b = ce(I1, J0), c = ce(I0, J1), d = ce(I1, J1);
    v.x += (R)0.25 * (((a.x + b.x) + c.x) + d.x);
    v.y += (R)0.25 * (((a.y + b.y) + c.y) + d.y);
    return v;
}

// Ascent of one level: the correction e2 + interpolation of the coarse iterate ec, the band
// sweeps around the hole, nu2 sweeps; T x T fine nodes go to e_out.  Only the tiles whose window
// meets the ring make the band sweeps, on a window 2 AN_BAND_SWEEPS nodes wider on every side
// (their values there are recomputed, the same, by the tiles that share them).  One launch for
// what were a prolongation (5 us), the band in one CTA (15) and a sweep launch (15-22):
// complex64 9 us at level 64, 10 at 128 and 256, 14 at 512, 28 at 1024, cold.
template <typename R, int T>
__global__ void __launch_bounds__(AN_TT, 2)
k_an_up(const typename CX<R>::T* __restrict__ e2, typename CX<R>::T* __restrict__ e_out,
        const typename CX<R>::T* __restrict__ rhs, AnGeo g, R h, R dinv, int nu2,
        const typename CX<R>::T* __restrict__ ec, int nc)
{
    typedef typename CX<R>::T c2;
    constexpr int AN_FT = T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = g.n, nt = (n + AN_FT) / AN_FT;
    const int i0 = (blockIdx.x / nt) * AN_FT, j0 = (blockIdx.x % nt) * AN_FT;
    const int h0 = 2 * nu2;
    const bool band = i0 - h0 <= g.b1 && i0 + AN_FT - 1 + h0 >= g.b0 && j0 - h0 <= g.b1 &&
                      j0 + AN_FT - 1 + h0 >= g.b0;
    const int skip = band ? 2 * AN_BAND_SWEEPS : 0;
    const int W = an_up_w(T, nu2, band), CW = W / 2 + 1;
    const AnWin<R> w = an_window<R>(smem_raw, i0 - h0 - skip, j0 - h0 - skip, W, W);
    c2* const Cs = w.R1 + W * (W >> 1);
    const int cy0 = w.y0 >> 1, cx0 = w.x0 >> 1;            // even origins
    pdl_wait();
    pdl_trigger();
    {
        const int Sc = nc + 1;
        const unsigned m = an_magic(CW);
        for (int q = threadIdx.x; q < CW * CW; q += AN_TT) {
            const int r = an_div(q, CW, m), I = cy0 + r, J = cx0 + (q - r * CW);
            const bool in = I >= 0 && I <= nc && J >= 0 && J <= nc;
            cp_async_elem<sizeof(c2)>(Cs + q, ec + (in ? (size_t)I * Sc + J : 0), in);
        }
    }
    an_stage<R>(w, W, W, e2, rhs, n, true);
    cp_async_wait_all();
    if constexpr (std::is_same<R, double>::value) {
        // Fixed point: in units of the window's largest value 2 after the correction, 4 after the
        // band (PDE rows: 1 / 2 a sweep), 13 / 2 after two sweeps (a row's sum 27: 2^58 * 27 <
        // 2^63), 9 after four (37, on 2^57)
        __shared__ int sx[AN_TT / 32];
        const FxH2 fp(h * h), fe(h);
        const bool plain = nu2 <= AN_FX_NU2 && fx_bits(dinv) == fx_bits(0.25);
        int ex = 0;
        if (plain) {
            ex = an_fx_exp(w, g, W, W, true, fp, fe);
            for (int q = threadIdx.x; q < CW * CW; q += AN_TT) ex = max(ex, fx_exp2(Cs[q]));
        }
        const int em = block_max_exp<AN_TT>(ex, sx) + (nu2 <= 2 ? 0 : 1);
        if (plain && fp.usable(em) && fe.usable(em)) {
            const AnWin<long long> f = an_fx_window(w, g, W, W, true, fp, fe, em);
            longlong2* const Fc = reinterpret_cast<longlong2*>(Cs);
            for (int q = threadIdx.x; q < CW * CW; q += AN_TT) Fc[q] = fx_q2(Cs[q], em);
            __syncthreads();
            const int ya = max(0, w.y0), yb = min(n, w.y0 + W - 1), xa = max(0, w.x0), xb = min(n, w.x0 + W - 1);
            const int nx = xb - xa + 1;
            const unsigned m = an_magic(nx);
            for (int q = threadIdx.x; q < nx * (yb - ya + 1); q += AN_TT) {
                const int r = an_div(q, nx, m), i = ya + r, j = xa + (q - r * nx);
                if (g.hole(i, j)) continue;
                const longlong2* p0 = Fc + ((i >> 1) - cy0) * CW, *p1 = Fc + (((i + 1) >> 1) - cy0) * CW;
                const int J0 = (j >> 1) - cx0, J1 = ((j + 1) >> 1) - cx0;
                const longlong2 a = p0[J0], b = p1[J0], c = p0[J1], d = p1[J1];
                longlong2* const p = f.E((i + j) & 1) + f.at(i, j);
                p->x += fx_shr<2>((a.x + b.x) + (c.x + d.x));
                p->y += fx_shr<2>((a.y + b.y) + (c.y + d.y));
            }
            __syncthreads();
            if (band)
                for (int k = 0; k < 2 * AN_BAND_SWEEPS; ++k) {
                    const int t = k + 1;
                    an_fx_half(f, g, max(g.b0, w.y0 + t), min(g.b1, w.y0 + W - 1 - t), max(g.b0, w.x0 + t),
                               min(g.b1, w.x0 + W - 1 - t), k & 1);
                    __syncthreads();
                }
            an_fx_sweeps(f, g, W, W, skip, nu2);
            const int S = n + 1;
            for (int q = threadIdx.x; q < AN_FT * AN_FT; q += AN_TT) {
                const int i = i0 + q / AN_FT, j = j0 + q % AN_FT;
                if (i <= n && j <= n) e_out[(size_t)i * S + j] = fx_d2(f.e(i, j), em);
            }
            return;
        }
    }
    __syncthreads();
    {
        const int ya = max(0, w.y0), yb = min(n, w.y0 + W - 1), xa = max(0, w.x0), xb = min(n, w.x0 + W - 1);
        // without band sweeps the first half-sweep overwrites colour 0 unread: colour 1 alone
        const bool half = !band && nu2 > 0;
        const int nx = half ? (xb - xa + 2) >> 1 : xb - xa + 1;
        const unsigned m = an_magic(nx);
        for (int q = threadIdx.x; q < nx * (yb - ya + 1); q += AN_TT) {
            const int r = an_div(q, nx, m), i = ya + r, u = q - r * nx;
            const int j = half ? xa + ((xa + i + 1) & 1) + 2 * u : xa + u;
            if (j > xb || g.hole(i, j)) continue;
            c2* const p = w.E((i + j) & 1) + w.at(i, j);
            *p = an_corrected<R>(*p, i, j, [&](int I, int J) -> c2 { return Cs[(I - cy0) * CW + (J - cx0)]; });
        }
    }
    __syncthreads();
    if (band) an_band_w<R>(w, g, W, W, false, h, dinv);
    an_sweeps_w<R>(w, g, W, W, skip, h, dinv, nu2);
    const int S = n + 1;
    for (int q = threadIdx.x; q < AN_FT * AN_FT; q += AN_TT) {
        const int i = i0 + q / AN_FT, j = j0 + q % AN_FT;
        if (i <= n && j <= n) e_out[(size_t)i * S + j] = w.e(i, j);
    }
}

// Coarsest level: e = Ainv rhs over its m unknowns (map: unknown -> node).  At holds Ainv
// transposed (column by column), so that neighbouring threads, which form neighbouring
// unknowns, read neighbouring words.  A warp's FP64 instruction holds its sub-core's pipe
// for 64 clocks: the columns are shared out so that every lane multiplies (a butterfly of
// FP64 adds per row took longer than the products), then each unknown adds its partial sums.
// part: room for AN_PARTS m complex FP64 sums.
constexpr int AN_PARTS = 14;
template <typename R, typename FR, typename FE>
__device__ __forceinline__ void an_dense_solve(const double* At, const int* __restrict__ map, int m, double2* part,
                                               FR rhs, FE put)
{
    const int groups = min(AN_PARTS, (int)blockDim.x / m), per = (m + groups - 1) / groups;
    const int gq = threadIdx.x / m, r = threadIdx.x - gq * m;
    if (gq < groups) {
        double ax = 0.0, ay = 0.0;
        for (int c = gq * per; c < min(m, (gq + 1) * per); ++c) {
            const double a = At[(size_t)c * m + r];
            const auto v = rhs(map[c]);
            ax = fma(a, an_widen(v.x), ax);
            ay = fma(a, an_widen(v.y), ay);
        }
        part[gq * m + r] = make_double2(ax, ay);
    }
    __syncthreads();
    // the two components of an unknown by two threads
    if ((int)threadIdx.x < 2 * m) {
        const int u = threadIdx.x >> 1;
        double s = 0.0;
        for (int k = 0; k < groups; ++k) s += (threadIdx.x & 1) ? part[k * m + u].y : part[k * m + u].x;
        put(map[u], threadIdx.x & 1, (R)s);
    }
}

// ---------------------------------------------------------------------------
// Coarse tail: the coarsest levels in one CTA, in shared memory
// ---------------------------------------------------------------------------
// The same V-cycle as the tile kernels (sweeps, restriction, prolongation, band sweeps,
// exact coarsest level), with block-wide barriers between its phases instead of kernel
// boundaries.  complex64 from 32 (1.6 K nodes with 16 and 8): a step of N = 64 takes 49 us, of
// N = 1024 192; from 64 (5.7 K nodes, whose 2 us half-sweeps one SM makes alone) 60 and 202, from
// 16 51 and 193.  FP64 from 16: one SM's FP64 rate makes the larger levels slower in one CTA
// than in tiles.  (From 64, 75 -> 47 us against rows by warps over type bytes and a butterfly
// per row of the dense solve.)
constexpr int AN_TAIL_TOP_F = 32;
constexpr int AN_TAIL_TOP_D = 16;
constexpr int AN_TAIL_MAX = 4;

template <typename R> struct AnTail {
    int L, nu1, nu2, load_e, m;
    R sigma;
    AnGeo geo[AN_TAIL_MAX];
    R h[AN_TAIL_MAX], dinv[AN_TAIL_MAX], ih2[AN_TAIL_MAX];       // (no conversions in the kernel)
    const double* At;
    const int* map;
};

// shared memory: per level the four planes ((n + 1) rows of n + 2), the top level's residual
// planes, the coarsest level's transposed inverse and partial sums
__host__ __device__ inline size_t an_tail_level(int n) { return (size_t)(n + 1) * (n + 2) * 2; }
template <typename R>
size_t an_tail_bytes(const int* ns, int L, int m)
{
    size_t c = (size_t)(ns[0] + 1) * (ns[0] + 2);
    for (int l = 0; l < L; ++l) c += an_tail_level(ns[l]);
    return an_a16(c * sizeof(typename CX<R>::T)) + an_a16((size_t)m * m * sizeof(double)) +
           (size_t)AN_PARTS * m * sizeof(double2);
}

template <typename R>
__global__ void __launch_bounds__(1024, 1)
k_an_tail(typename CX<R>::T* __restrict__ eg, const typename CX<R>::T* __restrict__ rg, AnTail<R> T)
{
    typedef typename CX<R>::T c2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c2* const base = reinterpret_cast<c2*>(smem_raw);
    // window l of the levels; the top level's residual planes follow the last one
    size_t off[AN_TAIL_MAX + 1];
    off[0] = 0;
#pragma unroll
    for (int l = 0; l < AN_TAIL_MAX; ++l) off[l + 1] = off[l] + (l < T.L ? an_tail_level(T.geo[l].n) : 0);
    const size_t c_end = off[AN_TAIL_MAX] + (size_t)(T.geo[0].n + 1) * (T.geo[0].n + 2);
    c2* const Res = base + off[AN_TAIL_MAX];
    double* const At = reinterpret_cast<double*>(smem_raw + an_a16(c_end * sizeof(c2)));
    double2* const part = reinterpret_cast<double2*>(smem_raw + an_a16(c_end * sizeof(c2)) +
                                                     an_a16((size_t)T.m * T.m * sizeof(double)));
    auto win = [&](int l) { return an_window<R>(base + off[l], 0, 0, T.geo[l].n + 1, T.geo[l].n + 2); };
    // the inverse arrives while the cycle descends (host-written: before the wait)
    for (int q = threadIdx.x; q < T.m * T.m; q += blockDim.x) cp_async_elem<8>(At + q, T.At + q, true);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    pdl_wait();
    pdl_trigger();
    {
        const int n = T.geo[0].n;
        const AnWin<R> w = win(0);
        an_stage<R>(w, n + 1, n + 1, eg, rg, n, T.load_e != 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // the coarse iterates start from zero
    {
        c2 z;
        z.x = 0;
        z.y = 0;
        for (int l = 1; l < T.L; ++l) {
            const int cnt = (T.geo[l].n + 1) * (T.geo[l].n + 2);        // both iterate planes
            for (int q = threadIdx.x; q < cnt; q += blockDim.x) base[off[l] + q] = z;
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    const R sig = T.sigma;
    // descent
    for (int l = 0; l + 1 < T.L; ++l) {
        const AnGeo g = T.geo[l], gc = T.geo[l + 1];
        const R h = T.h[l], dinv = T.dinv[l];
        const int n = g.n, W = n + 2;
        const AnWin<R> w = win(l);
        for (int k = 0; k < 2 * T.nu1; ++k) {
            an_half_w<R, false>(w, g, 0, n, 0, n, h, dinv, k & 1);
            __syncthreads();
        }
        const bool zero = T.nu1 == 0 && (l > 0 || !T.load_e);
        const R ih2 = T.ih2[l];
        const unsigned m = an_magic(n + 1);
        c2* const P[2] = {Res, Res + (n + 1) * (W >> 1)};
        for (int q = threadIdx.x; q < (n + 1) * (n + 1); q += blockDim.x) {
            const int i = an_div(q, n + 1, m), j = q - i * (n + 1);
            P[(i + j) & 1][w.at(i, j)] = an_resid_w<R>(w, g, i, j, h, ih2, sig, zero);
        }
        __syncthreads();
        const AnWin<R> wc = win(l + 1);
        const unsigned mc = an_magic(gc.n + 1);
        for (int q = threadIdx.x; q < (gc.n + 1) * (gc.n + 1); q += blockDim.x) {
            const int I = an_div(q, gc.n + 1, mc), J = q - I * (gc.n + 1);
            wc.Rh((I + J) & 1)[wc.at(I, J)] = an_restrict_node<R>(
                gc, I, J, [&](int i, int j) -> c2 { return P[(i + j) & 1][w.at(i, j)]; });
        }
        __syncthreads();
    }
    // the coarsest level, exactly
    {
        const AnWin<R> w = win(T.L - 1);
        const int S = T.geo[T.L - 1].n + 1;
        an_dense_solve<R>(
            At, T.map, T.m, part,
            [&](int q) -> c2 { const int i = q / S, j = q - i * S; return w.Rh((i + j) & 1)[w.at(i, j)]; },
            [&](int q, int im, R v) {
                const int i = q / S, j = q - i * S;
                c2* const p = w.E((i + j) & 1) + w.at(i, j);
                if (im) p->y = v;
                else p->x = v;
            });
        __syncthreads();
    }
    // ascent
    for (int l = T.L - 2; l >= 0; --l) {
        const AnGeo g = T.geo[l];
        const int n = g.n;
        const R h = T.h[l], dinv = T.dinv[l];
        const AnWin<R> w = win(l), wc = win(l + 1);
        const unsigned m = an_magic(n + 1);
        for (int q = threadIdx.x; q < (n + 1) * (n + 1); q += blockDim.x) {
            const int i = an_div(q, n + 1, m), j = q - i * (n + 1);
            if (g.hole(i, j)) continue;
            c2* const p = w.E((i + j) & 1) + w.at(i, j);
            *p = an_corrected<R>(*p, i, j, [&](int I, int J) -> c2 { return wc.e(I, J); });
        }
        __syncthreads();
        an_band_w<R>(w, g, n + 1, n + 1, true, h, dinv);
        for (int k = 0; k < 2 * T.nu2; ++k) {
            an_half_w<R, false>(w, g, 0, n, 0, n, h, dinv, k & 1);
            __syncthreads();
        }
    }
    {
        const AnWin<R> w = win(0);
        const int n = T.geo[0].n;
        const unsigned m = an_magic(n + 1);
        for (int q = threadIdx.x; q < (n + 1) * (n + 1); q += blockDim.x) {
            const int i = an_div(q, n + 1, m), j = q - i * (n + 1);
            eg[q] = w.e(i, j);
        }
    }
}

// Control of a solve, in device memory: its buffers (the step's graph is kept with the plan, the
// caller's pointers are not in it), the outer iteration's state, and the history's ring in
// page-locked memory.
struct AnCtl {
    double2* U[2];
    const double2* data;
    double* hist;                     // AN_HIST entries: step N at N % AN_HIST
    double tol, norm0, prev, rmin;
    int it, max_outer, run, status;   // status: AN_ACTIVE or the outcome
    int budget;                       // steps left of this launch
    unsigned ticket;
};
constexpr int AN_ACTIVE = 1000, AN_HIST = 4096;

// U := the hole data on hole nodes, 0 elsewhere (both iterate buffers); starts the control
__global__ void __launch_bounds__(AN_NT)
k_an_init(AnCtl* __restrict__ ctl, AnCtl c, const unsigned char* __restrict__ typ, long total)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *ctl = c;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const double2 v = (typ[t] == AN_HOLE) ? c.data[t] : make_double2(0.0, 0.0);
        c.U[0][t] = v;
        c.U[1][t] = v;
    }
}

// a further run of steps
__global__ void k_an_more(AnCtl* ctl, int budget) { ctl->budget = budget; }

// the result to the caller's buffer (U[0]), the outcome to the host
__global__ void __launch_bounds__(AN_NT)
k_an_fin(const AnCtl* __restrict__ ctl, int* __restrict__ out, long total)
{
    const int it = ctl->it;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[0] = it;
        out[1] = ctl->status;
    }
    if (!(it & 1) || ctl->status == AN_ACTIVE) return;
    double2* const u = ctl->U[0];
    const double2* const v = ctl->U[1];
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) u[t] = v[t];
}

// The last of a launch's blocks sums the np partials, applies the cavity's status rule and sets
// the loop's condition (gh != 0).  start: the start residual.
__device__ void an_finish(AnCtl* ctl, const double* part, int np, bool start, unsigned long long gh, double* sa)
{
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double r2 = 0.0;
    for (int b = threadIdx.x; b < np; b += blockDim.x) r2 += __ldcg(part + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if ((threadIdx.x & 31) == 0) sa[threadIdx.x >> 5] = r2;
    __syncthreads();
    if (threadIdx.x != 0) return;
    r2 = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) r2 += sa[w];
    AnCtl c = *ctl;
    c.ticket = 0u;
    const double norm = sqrt(r2);
    if (start) {
        c.norm0 = norm;
        c.hist[0] = norm == 0.0 ? 0.0 : 1.0;
        c.status = norm == 0.0 ? HELM_CONVERGED : !isfinite(norm) ? HELM_ENONFINITE : c.max_outer < 1 ? HELM_MAXITER
                                                                                                      : AN_ACTIVE;
    } else if (c.status == AN_ACTIVE) {            // (a solve that ended at its start: nothing)
        const double rel = norm / c.norm0;
        const int it = ++c.it;
        c.hist[it % AN_HIST] = rel;
        c.run = (rel >= c.prev) ? c.run + 1 : 0;
        c.prev = rel;
        c.rmin = fmin(c.rmin, rel);
        if (!isfinite(rel)) c.status = HELM_ENONFINITE;
        else if (rel <= c.tol) c.status = HELM_CONVERGED;
        else if (rel > 1e4 || (it >= 20 && c.run >= 10 && rel >= 2.0 * c.rmin)) c.status = HELM_DIVERGED;
        else if (it >= c.max_outer) c.status = HELM_MAXITER;
        --c.budget;
    }
    *ctl = c;
    if (gh) cudaGraphSetConditional((cudaGraphConditionalHandle)gh, c.status == AN_ACTIVE && c.budget > 0 ? 1u : 0u);
}

// part[block] = the block's sum (by warps in R, then in FP64)
template <typename R>
__device__ __forceinline__ void an_block_sum(R r2, double* sa, double* part)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if ((threadIdx.x & 31) == 0) sa[threadIdx.x >> 5] = (double)r2;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < AN_NT / 32; ++w) a += sa[w];
        part[blockIdx.x] = a;
    }
}

// An outer step's update and residual in one pass: U_out = U_in + e on the non-hole nodes (hole
// nodes keep the data in both buffers; e == nullptr: U_in as it is), r = b - B U_out in FP64
// (PDE: f - (Delta_h U + k^2 U); EDGE: q - (dU/dn - i k U)) into rhs, rounded to the inner
// precision; in FP64 also per-block sums of |r|^2 into part[b] (k_an_norm in complex64).
//
// A tile's T x T updated nodes and their ring go to shared memory, so that U is read once and
// e at all only here.  complex128: on the tile's fixed-point scale, the numerators being exact
// integer sums (6 FP64 operations a node instead of 16; an SM serves about 2 a clock); tiles
// outside the scale's range in FP64.  complex64 keeps the FP64 numerators, which bound it: an
// inner cycle in FP32 passes a residual that rounds otherwise in one node of a thousand on as
// 1e-10 .. 1e-9 of the next steps' residuals.  T as in an_tile; the grid strides over the tiles.
// 1024^2 complex64: 58 us in two launches -> 43 (36 at the start, without e), and 7 for the norm;
// its 16 FP64 operations a node take 29 us, its 64 bytes 9.  With the numerators in fixed point
// 28 us, for histories 3e-10 off.  1 / h^2 comes from the host: an FP64 division in every thread
// took 4 us.  256^2 complex128: a step 75 -> 73 us.
template <typename R, int T>
__global__ void __launch_bounds__(AN_NT)
k_an_step(AnCtl* ctl, const typename CX<R>::T* __restrict__ e, typename CX<R>::T* __restrict__ rhs, AnGeo g, int nt,
          double ih2, double ih, double k2, double k, double* part, unsigned long long gh)
{
    typedef typename CX<R>::T c2;
    constexpr int W = T + 2, PER = T * T / AN_NT;
    constexpr bool WIDE = std::is_same<R, double>::value;
    __shared__ longlong2 F[W * W];
    __shared__ int sx[AN_NT / 32];
    __shared__ double sa[AN_NT / 32];
    double2* const D = reinterpret_cast<double2*>(F);
    const int n = g.n, S = n + 1, tid = threadIdx.x;
    R r2 = 0;
    pdl_wait();
    pdl_trigger();
    const int par = ctl->it & 1;
    const double2* __restrict__ const Uin = ctl->U[par];
    double2* __restrict__ const Uout = ctl->U[par ^ 1];
    const double2* __restrict__ const data = ctl->data;
    for (int tile = blockIdx.x; tile < nt * nt; tile += gridDim.x) {
        const int ty = tile / nt, i0 = ty * T, j0 = (tile - ty * nt) * T;
        double2 c[PER], dv[PER], rv = make_double2(0.0, 0.0);
        int ex = 0, ro = -1;
        auto updated = [&](int i, int j, size_t q) {
            double2 v = Uin[q];
            if (e && !g.hole(i, j)) {
                const c2 ev = e[q];
                v.x += an_widen(ev.x);
                v.y += an_widen(ev.y);
            }
            if (WIDE) ex = max(ex, fx_exp2(v));
            return v;
        };
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int q = tid + p * AN_NT, i = i0 + q / T, j = j0 + q % T;
            c[p] = dv[p] = make_double2(0.0, 0.0);
            if (i > n || j > n) continue;
            const size_t gq = (size_t)i * S + j;
            c[p] = updated(i, j, gq);
            if (g.hole(i, j)) continue;
            dv[p] = data[gq];
            if (e) Uout[gq] = c[p];
        }
        if (tid < 4 * T + 4) {                    // the ring: two rows of W, two columns of T
            const int u = tid < 2 * W ? tid % W : (tid - 2 * W) % T + 1, b = tid < 2 * W ? tid / W : (tid - 2 * W) / T;
            const int ly = tid < 2 * W ? b * (W - 1) : u, lx = tid < 2 * W ? u : b * (W - 1);
            const int i = i0 - 1 + ly, j = j0 - 1 + lx;
            ro = ly * W + lx;
            if (i >= 0 && i <= n && j >= 0 && j <= n) rv = updated(i, j, (size_t)i * S + j);
        }
        int em = -1;                              // -1: FP64
        if constexpr (WIDE) {
            em = block_max_exp<AN_NT>(ex, sx);
            if (em == 0) em = FX_EMIN + 8;
            if (!fx_usable(em)) em = -1;
        } else {
            __syncthreads();                      // the last tile's readers are done
        }
        auto put = [&](int o, double2 v) {
            if (WIDE && em >= 0) F[o] = fx_q2(v, em);
            else D[o] = v;
        };
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int q = tid + p * AN_NT;
            put((q / T + 1) * W + q % T + 1, c[p]);
        }
        if (ro >= 0) put(ro, rv);
        __syncthreads();
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int q = tid + p * AN_NT, i = i0 + q / T, j = j0 + q % T, o = (q / T + 1) * W + q % T + 1;
            if (i > n || j > n || g.hole(i, j)) continue;
            const bool pde = !g.edge(i, j);
            const double2 cc = c[p];
            // an EDGE node's inward neighbours (o1; o2 = o1 but at a corner)
            const int o1 = i == 0 ? o + W : i == n ? o - W : j == 0 ? o + 1 : o - 1;
            const int o2 = (i == 0 || i == n) && (j == 0 || j == n) ? (j == 0 ? o + 1 : o - 1) : o1;
            double2 r;
            if (WIDE && em >= 0) {
                const longlong2 m = F[o];
                if (pde) {
                    const longlong2 a = F[o - W], b = F[o + W], l = F[o - 1], t = F[o + 1];
                    const long long sx2 = ((a.x + b.x) + (l.x + t.x)) - 4 * m.x, sy2 = ((a.y + b.y) + (l.y + t.y)) - 4 * m.y;
                    r.x = fma(fx_to_double(sx2, em), -ih2, fma(cc.x, -k2, dv[p].x));
                    r.y = fma(fx_to_double(sy2, em), -ih2, fma(cc.y, -k2, dv[p].y));
                } else {
                    const longlong2 a = F[o1], b = F[o2];
                    r.x = fma(fx_to_double(2 * m.x - (a.x + b.x), em), -0.5 * ih, fma(cc.y, -k, dv[p].x));
                    r.y = fma(fx_to_double(2 * m.y - (a.y + b.y), em), -0.5 * ih, fma(cc.x, k, dv[p].y));
                }
            } else if (pde) {
                const double2 a = D[o - W], b = D[o + W], l = D[o - 1], t = D[o + 1];
                r.x = dv[p].x - (((a.x + b.x) + (l.x + t.x) - 4.0 * cc.x) * ih2 + k2 * cc.x);
                r.y = dv[p].y - (((a.y + b.y) + (l.y + t.y) - 4.0 * cc.y) * ih2 + k2 * cc.y);
            } else {
                // dU/dn - i k U = (U - mean) / h + (k U.y, -k U.x)
                double2 m = D[o1];
                if (o2 != o1) m = make_double2((m.x + D[o2].x) * 0.5, (m.y + D[o2].y) * 0.5);
                r.x = dv[p].x - ((cc.x - m.x) * ih + k * cc.y);
                r.y = dv[p].y - ((cc.y - m.y) * ih - k * cc.x);
            }
            c2 ri;
            ri.x = an_narrow(r.x, R());
            ri.y = an_narrow(r.y, R());
            rhs[(size_t)i * S + j] = ri;
            if constexpr (WIDE) r2 += ri.x * ri.x + ri.y * ri.y;
        }
    }
    if constexpr (WIDE) {
        an_block_sum(r2, sa, part);
        an_finish(ctl, part, gridDim.x, e == nullptr, gh, sa);
    }
}

// per-block sums of |rhs|^2 of a complex64 step.  Its FP32 sums follow the rows, whatever the
// tiles: a start residual lives on a few nodes around the hole, and another order would move
// the history by their roundings (1e-9 of it).
__global__ void __launch_bounds__(AN_NT)
k_an_norm(const float2* __restrict__ rhs, AnGeo g, double* part, AnCtl* ctl, int start, unsigned long long gh)
{
    __shared__ double sa[AN_NT / 32];
    const int S = g.n + 1, total = S * S;
    float r2 = 0;
    pdl_wait();
    pdl_trigger();
    for (int t = blockIdx.x * AN_NT + threadIdx.x; t < total; t += gridDim.x * AN_NT) {
        const int i = t / S, j = t - i * S;
        if (g.hole(i, j)) continue;
        const float2 ri = rhs[t];
        r2 += ri.x * ri.x + ri.y * ri.y;
    }
    an_block_sum(r2, sa, part);
    an_finish(ctl, part, gridDim.x, start != 0, gh, sa);
}

// real part of U -> out (double), and min over PDE nodes of (-L + sqrt(L^2 + 4 E)) / (2 E)
// (positive doubles order as their bit patterns)
__global__ void __launch_bounds__(AN_NT)
k_an_real(const double2* __restrict__ U, double* __restrict__ out, long total)
{
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x)
        out[t] = U[t].x;
}

__global__ void __launch_bounds__(AN_NT)
k_an_kstar(const double* __restrict__ E, const double* __restrict__ L, const unsigned char* __restrict__ typ,
           long total, unsigned long long* __restrict__ out)
{
    double best = 1e300;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        if (typ[t] != AN_PDE) continue;
        const double e = E[t], l = L[t];
        if (!(e > 0.0)) continue;
        best = fmin(best, (-l + sqrt(l * l + 4.0 * e)) / (2.0 * e));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0 && best < 1e300) atomicMin(out, (unsigned long long)__double_as_longlong(best));
}


// ---- spectrum of G = A_sigma^{-1} M (Section 2.4's figure): M = -alpha on PDE rows, +i k
// on EDGE rows (M^H: -alpha, -i k) ----

__device__ __forceinline__ bool an_corner(int i, int j, int n)
{
    return (i == 0 || i == n) && (j == 0 || j == n);
}

// block sum of three doubles into part[3 b + 0..2]
__device__ __forceinline__ void an_sum3(double a, double b, double c, double* __restrict__ part)
{
    __shared__ double sm[3][AN_NT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sm[0][threadIdx.x >> 5] = a;
        sm[1][threadIdx.x >> 5] = b;
        sm[2][threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int w = 0; w < AN_NT / 32; ++w) t += sm[threadIdx.x][w];
        part[3 * blockIdx.x + threadIdx.x] = t;
    }
}

// rhs = s M x in the inner precision (hole rows 0)
template <typename R>
__global__ void __launch_bounds__(AN_NT)
k_an_mx(const double2* __restrict__ x, const unsigned char* __restrict__ typ, typename CX<R>::T* __restrict__ rhs,
        long total, double s, double alpha, double k)
{
    typedef typename CX<R>::T c2;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const unsigned char ty = typ[t];
        const double2 v = x[t];
        double rx = 0.0, ry = 0.0;
        if (ty == AN_PDE) {
            rx = -alpha * s * v.x;
            ry = -alpha * s * v.y;
        } else if (ty == AN_EDGE) {            // i k (v.x + i v.y)
            rx = -k * s * v.y;
            ry = k * s * v.x;
        }
        c2 r;
        r.x = an_narrow(rx, R());
        r.y = an_narrow(ry, R());
        rhs[t] = r;
    }
}

// power-iteration bookkeeping: sums of |e|^2 and of conj(x) e (re, im) per block, then x := e
template <typename R>
__global__ void __launch_bounds__(AN_NT)
k_an_pdot(double2* __restrict__ x, const typename CX<R>::T* __restrict__ e, const unsigned char* __restrict__ typ,
          long total, double* __restrict__ part)
{
    double a = 0.0, cr = 0.0, ci = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        if (typ[t] == AN_HOLE) {
            x[t] = make_double2(0.0, 0.0);
            continue;
        }
        const double ex = an_widen(e[t].x), ey = an_widen(e[t].y);
        const double2 xv = x[t];
        a += ex * ex + ey * ey;
        cr += xv.x * ex + xv.y * ey;
        ci += xv.x * ey - xv.y * ex;
        x[t] = make_double2(ex, ey);
    }
    an_sum3(a, cr, ci, part);
}

// Adjoint solve, first half.  With W = 1 on PDE rows and -1/h on EDGE rows, W A_sigma is
// symmetric once the corner rows and columns are dropped, and no other row references a
// corner; so A^{-T} y is: corners h y_c; the rest W A^{-1} W^{-1} (y + the corner rows'
// transposed couplings, +y_c / 2 on each corner's two inward neighbours), the solve taken
// with zero right-hand side at the corners.  This kernel forms that right-hand side from
// y = e, writes the corners' part of z = M^H A^{-T} y (-i k h y_c) into x, and sums |y|^2.
template <typename R>
__global__ void __launch_bounds__(AN_NT)
k_an_tprep(const typename CX<R>::T* __restrict__ e, typename CX<R>::T* __restrict__ rhs, double2* __restrict__ x,
           const unsigned char* __restrict__ typ, int n, double h, double k, double* __restrict__ part)
{
    typedef typename CX<R>::T c2;
    const int S = n + 1;
    const long total = (long)S * S;
    double a = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const unsigned char ty = typ[t];
        c2 r;
        r.x = 0;
        r.y = 0;
        if (ty == AN_HOLE) {
            rhs[t] = r;
            x[t] = make_double2(0.0, 0.0);
            continue;
        }
        const int q = (int)t, i = q / S, j = q % S;
        double yx = an_widen(e[q].x), yy = an_widen(e[q].y);
        a += yx * yx + yy * yy;
        if (an_corner(i, j, n)) {
            rhs[q] = r;
            x[q] = make_double2(k * h * yy, -k * h * yx);     // -i k h y_c
            continue;
        }
        if (ty == AN_EDGE) {
            if ((j == 0 || j == n) && (i == 1 || i == n - 1)) {
                const c2 c = e[(i == 1 ? 0 : n) * S + j];
                yx += 0.5 * an_widen(c.x);
                yy += 0.5 * an_widen(c.y);
            }
            if ((i == 0 || i == n) && (j == 1 || j == n - 1)) {
                const c2 c = e[i * S + (j == 1 ? 0 : n)];
                yx += 0.5 * an_widen(c.x);
                yy += 0.5 * an_widen(c.y);
            }
            yx *= -h;
            yy *= -h;
        }
        r.x = an_narrow(yx, R());
        r.y = an_narrow(yy, R());
        rhs[q] = r;
    }
    an_sum3(a, 0.0, 0.0, part);
}

// Adjoint solve, second half: z = M^H W s off the corners (PDE: -alpha s; EDGE: (-i k) (-s / h)
// = (i k / h) s) into x; sums |z|^2 over every node (the corners' z from k_an_tprep)
template <typename R>
__global__ void __launch_bounds__(AN_NT)
k_an_tfin(const typename CX<R>::T* __restrict__ e, double2* __restrict__ x, const unsigned char* __restrict__ typ,
          int n, double h, double alpha, double k, double* __restrict__ part)
{
    const int S = n + 1;
    const long total = (long)S * S;
    double a = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const unsigned char ty = typ[t];
        if (ty == AN_HOLE) continue;
        const int q = (int)t, i = q / S, j = q % S;
        double2 z;
        if (an_corner(i, j, n)) {
            z = x[q];
        } else {
            const double sx = an_widen(e[q].x), sy = an_widen(e[q].y);
            if (ty == AN_PDE) {
                z.x = -alpha * sx;
                z.y = -alpha * sy;
            } else {
                z.x = -k / h * sy;
                z.y = k / h * sx;
            }
            x[q] = z;
        }
        a += z.x * z.x + z.y * z.y;
    }
    an_sum3(a, 0.0, 0.0, part);
}

// Lanczos on the real symmetric K = A^T D A, D = diag(1 / alpha^2 on PDE rows, 1 / k^2 on EDGE
// rows) = (G^{-1})^H G^{-1}: its largest eigenvalue is 1 / sigma_min(G)^2.  y = D A v:
__global__ void __launch_bounds__(AN_NT)
k_an_lz_a(const double* __restrict__ v, double* __restrict__ y, const unsigned char* __restrict__ typ, int n,
          double h, double sigma, double dp, double de)
{
    const int S = n + 1;
    const long total = (long)S * S;
    const double ih2 = 1.0 / (h * h), ih = 1.0 / h;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const unsigned char ty = typ[t];
        const int q = (int)t, i = q / S, j = q % S;
        double r = 0.0;
        if (ty == AN_PDE) {
            // hole entries of v are zero
            r = (((v[q - S] + v[q + S]) + (v[q - 1] + v[q + 1])) - 4.0 * v[q]) * ih2 - sigma * v[q];
            r *= dp;
        } else if (ty == AN_EDGE) {
            double m = 0.0;
            int c = 0;
            if (i == 0) { m += v[S + j]; ++c; }
            if (i == n) { m += v[(n - 1) * S + j]; ++c; }
            if (j == 0) { m += v[i * S + 1]; ++c; }
            if (j == n) { m += v[i * S + n - 1]; ++c; }
            if (c == 2) m *= 0.5;
            r = (v[q] - m) * ih * de;
        }
        y[q] = r;
    }
}

// w = A^T y - beta v_prev (A^T gathered: PDE column j: its own row, its PDE neighbours'
// rows (1/h^2) and its EDGE neighbours' rows (-1/h, j being their inward neighbour); EDGE
// column: its own row (1/h), its inward neighbour's row (1/h^2), and the rows of the
// corners whose inward neighbour it is (-1/(2h)); corner column: its own row (1/h));
// part[3 b] = sum v . w
__global__ void __launch_bounds__(AN_NT)
k_an_lz_at(const double* __restrict__ y, const double* __restrict__ v, const double* __restrict__ vp, double beta,
           double* __restrict__ w, const unsigned char* __restrict__ typ, int n, double h, double sigma,
           double* __restrict__ part)
{
    const int S = n + 1;
    const long total = (long)S * S;
    const double ih2 = 1.0 / (h * h), ih = 1.0 / h;
    double a = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const unsigned char ty = typ[t];
        const int q = (int)t, i = q / S, j = q % S;
        double r = 0.0;
        if (ty == AN_PDE) {
            r = (-4.0 * ih2 - sigma) * y[q];
            const int nb[4] = {q - S, q + S, q - 1, q + 1};
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const unsigned char tn = typ[nb[d]];
                if (tn == AN_PDE) r += ih2 * y[nb[d]];
                else if (tn == AN_EDGE) r -= ih * y[nb[d]];
            }
        } else if (ty == AN_EDGE) {
            r = ih * y[q];
            if (!an_corner(i, j, n)) {
                const int in = (i == 0) ? S + j : (i == n) ? (n - 1) * S + j : (j == 0) ? i * S + 1 : i * S + n - 1;
                r += ih2 * y[in];
                if ((j == 0 || j == n) && (i == 1 || i == n - 1)) r -= 0.5 * ih * y[(i == 1 ? 0 : n) * S + j];
                if ((i == 0 || i == n) && (j == 1 || j == n - 1)) r -= 0.5 * ih * y[i * S + (j == 1 ? 0 : n)];
            }
        }
        r -= beta * vp[q];
        w[q] = r;
        a += v[q] * r;
    }
    an_sum3(a, 0.0, 0.0, part);
}

// w -= a v, part[3 b] = sum w^2
__global__ void __launch_bounds__(AN_NT)
k_an_lz_orth(double* __restrict__ w, const double* __restrict__ v, double a, long total, double* __restrict__ part)
{
    double s = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const double r = w[t] - a * v[t];
        w[t] = r;
        s += r * r;
    }
    an_sum3(s, 0.0, 0.0, part);
}

// v = s w; a seeded start vector when w == nullptr (hole nodes 0); part[3 b] = sum v^2
__global__ void __launch_bounds__(AN_NT)
k_an_lz_scale(double* __restrict__ v, const double* __restrict__ w, double s, const unsigned char* __restrict__ typ,
              long total, double* __restrict__ part)
{
    double a = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        double r;
        if (w) {
            r = s * w[t];
        } else {
            unsigned long long z = 0x9e3779b97f4a7c15ull * (unsigned long long)(t + 1);
            z = (z ^ (z >> 31)) * 0xbf58476d1ce4e5b9ull;
            z ^= z >> 29;
            r = (typ[t] == AN_HOLE) ? 0.0 : ((double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5);
        }
        v[t] = r;
        a += r * r;
    }
    an_sum3(a, 0.0, 0.0, part);
}

// complex seeded start vector (hole 0) into x; part: sums of |x|^2
__global__ void __launch_bounds__(AN_NT)
k_an_seed(double2* __restrict__ x, const unsigned char* __restrict__ typ, long total, double* __restrict__ part)
{
    double a = 0.0;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        unsigned long long z = 0xd1b54a32d192ed03ull * (unsigned long long)(t + 7);
        z = (z ^ (z >> 31)) * 0xbf58476d1ce4e5b9ull;
        z ^= z >> 29;
        const double re = (double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
        z ^= z >> 31;
        const double im = (double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5;
        const double2 v = (typ[t] == AN_HOLE) ? make_double2(0.0, 0.0) : make_double2(re, im);
        x[t] = v;
        a += v.x * v.x + v.y * v.y;
    }
    an_sum3(a, 0.0, 0.0, part);
}

}  // namespace
}  // namespace helm

using namespace helm;

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct helm_annulus {
    int N = 0, prec = HELM_PREC_MIXED;
    double side = 1.0, hole = 0.15, k = 0.0, alpha = 0.0, sigma = 0.0;
    int nu1 = 2, nu2 = 2, cycles = 1;
    struct Level {
        int n;
        double h;
        unsigned char* typ;
        void* e;
        void* rhs;
        void* e2;                         // the swept iterate between descent and ascent
        int b0, b1, lo, hi;               // band ring [b0, b1]^2 minus the hole box [lo, hi]^2
    };
    std::vector<Level> lev;
    double* At = nullptr;                 // the coarsest level's inverse, transposed
    int* map = nullptr;
    int m = 0;
    double2* U1 = nullptr;
    double* part = nullptr;
    AnCtl* ctl = nullptr;
    double* h_hist = nullptr;             // page-locked: the history's ring, the outcome behind it
    cudaGraphExec_t loop = nullptr;       // outer steps until the control says otherwise
    uint64_t loop_step = 0;               // kernels of one of them
    int nblk = 0;
    unsigned long long* kmin = nullptr;
    cudaStream_t stream = nullptr;
    std::vector<void*> allocs;
    cudaStream_t ls = nullptr;            // where an_vcycle and the step launch (stream, or cap)
    cudaStream_t cap = nullptr;           // non-blocking stream for capturing the loop's body
    bool capturing = false;
    uint64_t captured = 0;                // kernels recorded by the capture in progress
    int t0 = -1;                          // first level of the one-CTA coarse tail
    size_t tail_bytes = 0;
};

namespace {

#define AN_CK(call)                                                                             \
    do {                                                                                        \
        cudaError_t _e = (call);                                                                \
        if (_e != cudaSuccess) {                                                                \
            char _b[200];                                                                       \
            snprintf(_b, sizeof _b, "%s: %s", #call, cudaGetErrorString(_e));                   \
            note_error(_b);                                                                     \
            return HELM_ECUDA;                                                                  \
        }                                                                                       \
    } while (0)

// node types of a level (the oracle's rule: closed hole, outer edge rows elsewhere)
std::vector<unsigned char> an_types(int n, double side, double hole)
{
    const double h = side / n, eps = 1e-9 * side;
    std::vector<unsigned char> t((size_t)(n + 1) * (n + 1), AN_PDE);
    for (int i = 0; i <= n; ++i)
        for (int j = 0; j <= n; ++j) {
            const double x = -0.5 * side + i * h, y = -0.5 * side + j * h;
            unsigned char v = AN_PDE;
            if (i == 0 || i == n || j == 0 || j == n) v = AN_EDGE;
            if (std::fabs(x) <= hole + eps && std::fabs(y) <= hole + eps) v = AN_HOLE;
            t[(size_t)i * (n + 1) + j] = v;
        }
    return t;
}

bool an_geometry_ok(const std::vector<unsigned char>& t, int n)
{
    bool any = false;
    for (int i = 0; i <= n; ++i)
        for (int j = 0; j <= n; ++j) {
            const bool hole = t[(size_t)i * (n + 1) + j] == AN_HOLE;
            any |= hole;
            if (hole && (i <= 1 || i >= n - 1 || j <= 1 || j >= n - 1)) return false;
        }
    return any;
}

// dense inverse of the coarsest level's A_sigma on its unknowns (Gauss-Jordan, partial pivots)
bool an_coarse_inverse(const std::vector<unsigned char>& t, int n, double h, double sigma,
                       std::vector<double>& inv, std::vector<int>& map)
{
    const int S = n + 1;
    std::vector<int> idx((size_t)S * S, -1);
    map.clear();
    for (int q = 0; q < S * S; ++q)
        if (t[q] != AN_HOLE) { idx[q] = (int)map.size(); map.push_back(q); }
    const int m = (int)map.size();
    std::vector<double> A((size_t)m * m, 0.0);
    for (int r = 0; r < m; ++r) {
        const int q = map[r], i = q / S, j = q % S;
        if (t[q] == AN_PDE) {
            A[(size_t)r * m + r] = -4.0 / (h * h) - sigma;
            const int nb[4] = {q - S, q + S, q - 1, q + 1};
            for (int c : nb)
                if (idx[c] >= 0) A[(size_t)r * m + idx[c]] += 1.0 / (h * h);
        } else {
            std::vector<int> in;
            if (i == 0) in.push_back(q + S);
            if (i == n) in.push_back(q - S);
            if (j == 0) in.push_back(q + 1);
            if (j == n) in.push_back(q - 1);
            A[(size_t)r * m + r] = 1.0 / h;
            for (int c : in) A[(size_t)r * m + idx[c]] -= 1.0 / (h * in.size());
        }
    }
    inv.assign((size_t)m * m, 0.0);
    for (int r = 0; r < m; ++r) inv[(size_t)r * m + r] = 1.0;
    for (int c = 0; c < m; ++c) {
        int p = c;
        for (int r = c + 1; r < m; ++r)
            if (std::fabs(A[(size_t)r * m + c]) > std::fabs(A[(size_t)p * m + c])) p = r;
        if (std::fabs(A[(size_t)p * m + c]) < 1e-300) return false;
        if (p != c)
            for (int k = 0; k < m; ++k) {
                std::swap(A[(size_t)p * m + k], A[(size_t)c * m + k]);
                std::swap(inv[(size_t)p * m + k], inv[(size_t)c * m + k]);
            }
        const double d = A[(size_t)c * m + c];
        for (int k = 0; k < m; ++k) {
            A[(size_t)c * m + k] /= d;
            inv[(size_t)c * m + k] /= d;
        }
        for (int r = 0; r < m; ++r) {
            if (r == c) continue;
            const double f = A[(size_t)r * m + c];
            if (f == 0.0) continue;
            for (int k = 0; k < m; ++k) {
                A[(size_t)r * m + k] -= f * A[(size_t)c * m + k];
                inv[(size_t)r * m + k] -= f * inv[(size_t)c * m + k];
            }
        }
    }
    return true;
}

// every shared-memory size the kernels of a plan can ask for (any nu1, nu2 <= 8)
template <typename R>
cudaError_t an_attrs()
{
    auto set = [](auto* k, size_t b) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
    };
    cudaError_t e = set(k_an_down<R, 32>, an_down_bytes<R>(32, 8));
    if (e == cudaSuccess) e = set(k_an_down<R, 16>, an_down_bytes<R>(16, 8));
    if (e == cudaSuccess) e = set(k_an_up<R, 32>, an_up_bytes<R>(32, 8));
    if (e == cudaSuccess) e = set(k_an_up<R, 16>, an_up_bytes<R>(16, 8));
    if (e == cudaSuccess) e = set(k_an_tail<R>, AN_SMEM_MAX);
    return e;
}

// kernels launched (or recorded into a step graph, counted at each replay)
void an_count(helm_annulus* a, uint64_t n)
{
    if (a->capturing) a->captured += n;
    else add_launches(n);
}

AnGeo an_geo(const helm_annulus::Level& L) { return AnGeo{L.n, L.lo, L.hi, L.b0, L.b1}; }

// fine nodes per side of a tile: the smaller tiles where the larger would not reach every SM
// (each is then bound by its own phases, in FP64 by one SM's FP64 rate: N = 256 FP64 9.9 ms a
// solve with 32 everywhere, 6.0 with this rule; 512 complex64 4.1 -> 3.8)
int an_tile(int n)
{
    const int nt = (n + 32) / 32;
    return nt * nt >= 152 ? 32 : 16;
}

template <typename R, int T>
helm_status an_down(helm_annulus* a, const helm_annulus::Level& L, const helm_annulus::Level& C, bool zero)
{
    typedef typename CX<R>::T c2;
    const R h = (R)L.h, dinv = (R)(1.0 / (4.0 + a->sigma * L.h * L.h));
    const int nt = (C.n + T / 2) / (T / 2);
    AN_CK(launch_k(k_an_down<R, T>, dim3(nt * nt), dim3(AN_TT), an_down_bytes<R>(T, a->nu1), a->ls, (const c2*)L.e,
                   (c2*)L.e2, (const c2*)L.rhs, an_geo(L), h, dinv, (R)a->sigma, (R)1 / (h * h), a->nu1, zero ? 0 : 1,
                   (c2*)C.rhs, an_geo(C)));
    an_count(a, 1);
    return HELM_OK;
}

template <typename R, int T>
helm_status an_up(helm_annulus* a, const helm_annulus::Level& L, const helm_annulus::Level& C)
{
    typedef typename CX<R>::T c2;
    const R h = (R)L.h, dinv = (R)(1.0 / (4.0 + a->sigma * L.h * L.h));
    const int nt = (L.n + T) / T;
    AN_CK(launch_k(k_an_up<R, T>, dim3(nt * nt), dim3(AN_TT), an_up_bytes<R>(T, a->nu2), a->ls, (const c2*)L.e2,
                   (c2*)L.e, (const c2*)L.rhs, an_geo(L), h, dinv, a->nu2, (const c2*)C.e, C.n));
    an_count(a, 1);
    return HELM_OK;
}

// One V(nu1, nu2) cycle from level l down.  The iterate goes e -> e2 (descent), then e2 + the
// coarse correction -> e (ascent): the tiles of a launch stage windows of the buffer that
// none of them writes.
template <typename R>
helm_status an_vcycle(helm_annulus* a, int l, bool zero)
{
    typedef typename CX<R>::T c2;
    const auto& L = a->lev[l];
    cudaStream_t s = a->ls;
    if (l == a->t0) {                      // this level and all coarser ones in one CTA
        AnTail<R> T{};
        T.L = (int)a->lev.size() - l;
        T.nu1 = a->nu1;
        T.nu2 = a->nu2;
        T.load_e = zero ? 0 : 1;
        T.m = a->m;
        T.sigma = (R)a->sigma;
        T.At = a->At;
        T.map = a->map;
        for (int i = 0; i < T.L; ++i) {
            const auto& V = a->lev[l + i];
            T.geo[i] = an_geo(V);
            T.h[i] = (R)V.h;
            T.dinv[i] = (R)(1.0 / (4.0 + a->sigma * V.h * V.h));
            T.ih2[i] = (R)1 / ((R)V.h * (R)V.h);
        }
        for (int i = T.L; i < AN_TAIL_MAX; ++i) T.geo[i] = AnGeo{0, 0, 0, 0, 0};
        AN_CK(launch_k(k_an_tail<R>, dim3(1), dim3(1024), a->tail_bytes, s, (c2*)L.e, (const c2*)L.rhs, T));
        an_count(a, 1);
        return HELM_OK;
    }
    const auto& C = a->lev[l + 1];
    helm_status st = an_tile(L.n) == 32 ? an_down<R, 32>(a, L, C, zero) : an_down<R, 16>(a, L, C, zero);
    if (st != HELM_OK) return st;
    st = an_vcycle<R>(a, l + 1, true);
    if (st != HELM_OK) return st;
    return an_tile(L.n) == 32 ? an_up<R, 32>(a, L, C) : an_up<R, 16>(a, L, C);
}

// The update and residual of a step on a->ls (start: the start residual); cond: the handle of the
// loop that it ends (0: none).
template <typename R>
helm_status an_step(helm_annulus* a, bool start, unsigned long long cond)
{
    typedef typename CX<R>::T c2;
    const auto& L0 = a->lev[0];
    const int T = an_tile(a->N), nt = (a->N + T) / T;
    auto launch = [&](auto* kern) {
        return launch_k(kern, dim3(std::min(nt * nt, a->nblk)), dim3(AN_NT), (size_t)0, a->ls, a->ctl,
                        start ? (const c2*)nullptr : (const c2*)L0.e, (c2*)L0.rhs, an_geo(L0), nt,
                        1.0 / (L0.h * L0.h), 1.0 / L0.h, a->k * a->k, a->k, a->part, cond);
    };
    AN_CK(T == 32 ? launch(k_an_step<R, 32>) : launch(k_an_step<R, 16>));
    an_count(a, 1);
    if constexpr (std::is_same<R, float>::value) {
        AN_CK(launch_k(k_an_norm, dim3(a->nblk), dim3(AN_NT), (size_t)0, a->ls, (const c2*)L0.rhs, an_geo(L0),
                       a->part, a->ctl, start ? 1 : 0, cond));
        an_count(a, 1);
    }
    return HELM_OK;
}

template <typename R>
helm_status an_outer(helm_annulus* a, unsigned long long cond)
{
    for (int c = 0; c < a->cycles; ++c) {
        const helm_status st = an_vcycle<R>(a, 0, c == 0);
        if (st != HELM_OK) return st;
    }
    return an_step<R>(a, false, cond);
}

void an_drop_loop(helm_annulus* a)
{
    if (a->loop) cudaGraphExecDestroy(a->loop);
    a->loop = nullptr;
}

// The outer steps as one graph: a WHILE node whose body is a step (its parameters change with
// the plan's cycle and shift alone).  Left unset where the graph cannot be built.
// The host saw every step's partial norms before: 1024^2 complex64 10.61 -> 10.37 ms,
// 256^2 complex128 3.89 -> 3.61 ms, two graphs built in each solve included.
template <typename R>
void an_build_loop(helm_annulus* a)
{
    cudaGraph_t g = nullptr, got = nullptr;
    if (cudaGraphCreate(&g, 0) != cudaSuccess) { cudaGetLastError(); return; }
    cudaGraphConditionalHandle cond = 0;
    cudaGraphNodeParams p = {cudaGraphNodeTypeConditional};
    cudaGraphNode_t node;
    bool ok = cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
    if (ok) {
        p.conditional.handle = cond;
        p.conditional.type = cudaGraphCondTypeWhile;
        p.conditional.size = 1;
        ok = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &p) == cudaSuccess;
    }
    if (ok && cudaStreamBeginCaptureToGraph(a->cap, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                            cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        const cudaStream_t s = a->ls;
        a->ls = a->cap;
        a->capturing = true;
        a->captured = 0;
        const helm_status st = an_outer<R>(a, (unsigned long long)cond);
        a->capturing = false;
        a->ls = s;
        ok = cudaStreamEndCapture(a->cap, &got) == cudaSuccess && st == HELM_OK &&
             cudaGraphInstantiate(&a->loop, g, 0) == cudaSuccess;
        a->loop_step = a->captured;
        if (!ok) a->loop = nullptr;
    }
    cudaGraphDestroy(g);
    cudaGetLastError();
}

template <typename R>
helm_status an_solve(helm_annulus* a, const double2* data, double2* u, double tol, int max_outer, int* iters,
                     double* hist, int* final_status)
{
    cudaStream_t s = a->stream;
    a->ls = s;
    const long total = (long)(a->N + 1) * (a->N + 1);
    if (!a->loop && max_outer > 0) an_build_loop<R>(a);
    AnCtl c{};
    c.U[0] = u;
    c.U[1] = a->U1;
    c.data = data;
    c.hist = a->h_hist;
    c.tol = tol;
    c.prev = c.rmin = 1.0;
    c.max_outer = max_outer;
    c.status = AN_ACTIVE;
    c.budget = AN_HIST - 1;
    volatile int* const out = reinterpret_cast<int*>(a->h_hist + AN_HIST);
    k_an_init<<<grid_for(total), AN_NT, 0, s>>>(a->ctl, c, a->lev[0].typ, total);
    add_launches(1);
    // start: r_0 = b from U[0] (the hole data, zero elsewhere)
    helm_status st = an_step<R>(a, true, 0);
    if (st != HELM_OK) return st;
    // rounds of up to AN_HIST - 1 steps (the ring holds a round's history); without a graph a
    // step each
    for (int done = -1;;) {
        if (max_outer > 0 && a->loop) AN_CK(cudaGraphLaunch(a->loop, s));
        else if (max_outer > 0 && (st = an_outer<R>(a, 0)) != HELM_OK) return st;
        k_an_fin<<<grid_for(total), AN_NT, 0, s>>>(a->ctl, const_cast<int*>(out), total);
        AN_CK(cudaGetLastError());
        AN_CK(cudaStreamSynchronize(s));
        const int it = out[0];
        if (a->loop) add_launches(a->loop_step * (uint64_t)(it - std::max(done, 0)));
        add_launches(1);
        for (int q = done + 1; hist && q <= it; ++q) hist[q] = a->h_hist[q % AN_HIST];
        done = it;
        if (out[1] != AN_ACTIVE) {
            if (iters) *iters = it;
            *final_status = out[1];
            return HELM_OK;
        }
        k_an_more<<<1, 1, 0, s>>>(a->ctl, AN_HIST - 1);
        add_launches(1);
    }
}


// ---- spectrum of G (Section 2.4's figure) ----

// e := A_sigma^{-1} rhs on level 0 by `cycles` multigrid cycles from zero
template <typename R>
helm_status an_apply_inv(helm_annulus* a, int cycles)
{
    typedef typename CX<R>::T c2;
    const auto& L0 = a->lev[0];
    const long total = (long)(a->N + 1) * (a->N + 1);
    a->ls = a->stream;
    for (int c = 0; c < cycles; ++c) {
        const helm_status st = an_vcycle<R>(a, 0, c == 0);
        if (st != HELM_OK) return st;
    }
    return HELM_OK;
}

// per-call reduction buffers (three doubles per block) and their host copy
struct AnSums {
    double* d = nullptr;
    double* h = nullptr;
    int nb = 0;
    ~AnSums()
    {
        if (d) cudaFree(d);
        if (h) cudaFreeHost(h);
    }
    helm_status init(int nblk)
    {
        nb = nblk;
        if (cudaMalloc(&d, 3 * sizeof(double) * nb) != cudaSuccess) return HELM_ENOMEM;
        if (cudaMallocHost(&h, 3 * sizeof(double) * nb) != cudaSuccess) return HELM_ENOMEM;
        return HELM_OK;
    }
    // block sums -> out[0..2] (fixed order)
    helm_status fetch(cudaStream_t s, double* out)
    {
        AN_CK(cudaMemcpyAsync(h, d, 3 * sizeof(double) * nb, cudaMemcpyDeviceToHost, s));
        AN_CK(cudaStreamSynchronize(s));
        out[0] = out[1] = out[2] = 0.0;
        for (int b = 0; b < nb; ++b)
            for (int c = 0; c < 3; ++c) out[c] += h[3 * b + c];
        return HELM_OK;
    }
};

// Power iteration x <- G x / ||G x||: rho ~ ||G x|| (||x|| = 1), lambda ~ x^H G x.
template <typename R>
helm_status an_spectral(helm_annulus* a, int max_iter, double tol, int cycles, double* rho, double* lre,
                        double* lim, int* iters, bool* conv)
{
    typedef typename CX<R>::T c2;
    const auto& L0 = a->lev[0];
    const long total = (long)(a->N + 1) * (a->N + 1);
    cudaStream_t s = a->stream;
    AnSums sums;
    helm_status st = sums.init(a->nblk);
    if (st != HELM_OK) return st;
    double v[3];
    k_an_seed<<<a->nblk, AN_NT, 0, s>>>(a->U1, L0.typ, total, sums.d);
    an_count(a, 1);
    if ((st = sums.fetch(s, v)) != HELM_OK) return st;
    double sc = 1.0 / std::sqrt(v[0]), prev = 0.0, r = 0.0;
    int ok = 0, it = 0;
    *conv = false;
    for (it = 1; it <= max_iter; ++it) {
        k_an_mx<R><<<a->nblk, AN_NT, 0, s>>>(a->U1, L0.typ, (c2*)L0.rhs, total, sc, a->alpha, a->k);
        an_count(a, 1);
        if ((st = an_apply_inv<R>(a, cycles)) != HELM_OK) return st;
        k_an_pdot<R><<<a->nblk, AN_NT, 0, s>>>(a->U1, (const c2*)L0.e, L0.typ, total, sums.d);
        an_count(a, 1);
        AN_CK(cudaGetLastError());
        if ((st = sums.fetch(s, v)) != HELM_OK) return st;
        r = std::sqrt(v[0]);
        *lre = sc * v[1];
        *lim = sc * v[2];
        if (!(r > 0.0) || !std::isfinite(r)) return HELM_ENONFINITE;
        sc = 1.0 / r;
        ok = (std::fabs(r - prev) <= tol * r) ? ok + 1 : 0;
        prev = r;
        if (ok >= 2) {
            *conv = true;
            break;
        }
    }
    *rho = r;
    *iters = std::min(it, max_iter);
    return HELM_OK;
}

// largest eigenvalue of the symmetric tridiagonal matrix (diag a[0..m-1], off-diagonal
// b[1..m-1]) by bisection on the Sturm count
double tridiag_max(const std::vector<double>& a, const std::vector<double>& b, int m)
{
    double lo = 1e300, hi = -1e300;
    for (int i = 0; i < m; ++i) {
        const double r = (i > 0 ? std::fabs(b[i]) : 0.0) + (i + 1 < m ? std::fabs(b[i + 1]) : 0.0);
        lo = std::min(lo, a[i] - r);
        hi = std::max(hi, a[i] + r);
    }
    auto below = [&](double x) {                  // eigenvalues < x
        int c = 0;
        double d = 1.0;
        for (int i = 0; i < m; ++i) {
            d = a[i] - x - (i > 0 ? b[i] * b[i] / d : 0.0);
            if (d == 0.0) d = -1e-300;
            if (d < 0.0) ++c;
        }
        return c;
    };
    for (int k = 0; k < 200 && hi - lo > 1e-15 * std::max(std::fabs(lo), std::fabs(hi)); ++k) {
        const double mid = 0.5 * (lo + hi);
        if (below(mid) >= m) hi = mid;
        else lo = mid;
    }
    return 0.5 * (lo + hi);
}

// sigma_max(G) by power iteration on G^H G (adjoint solves through the symmetrised
// operator), sigma_min(G) = 1 / sqrt(lambda_max(A^T D A)) by Lanczos (no solves).
template <typename R>
helm_status an_singular(helm_annulus* a, int max_iter, double tol, int cycles, double* smax, double* smin,
                        int* iters, bool* conv)
{
    typedef typename CX<R>::T c2;
    const auto& L0 = a->lev[0];
    const int n = a->N;
    const long total = (long)(n + 1) * (n + 1);
    cudaStream_t s = a->stream;
    AnSums sums;
    helm_status st = sums.init(a->nblk);
    if (st != HELM_OK) return st;
    double v[3];
    // sigma_max
    k_an_seed<<<a->nblk, AN_NT, 0, s>>>(a->U1, L0.typ, total, sums.d);
    an_count(a, 1);
    if ((st = sums.fetch(s, v)) != HELM_OK) return st;
    double sc = 1.0 / std::sqrt(v[0]), prev = 0.0, est = 0.0;
    int ok = 0, it1 = 0;
    bool c1 = false;
    for (it1 = 1; it1 <= max_iter; ++it1) {
        k_an_mx<R><<<a->nblk, AN_NT, 0, s>>>(a->U1, L0.typ, (c2*)L0.rhs, total, sc, a->alpha, a->k);
        an_count(a, 1);
        if ((st = an_apply_inv<R>(a, cycles)) != HELM_OK) return st;
        k_an_tprep<R><<<a->nblk, AN_NT, 0, s>>>((const c2*)L0.e, (c2*)L0.rhs, a->U1, L0.typ, n, L0.h, a->k, sums.d);
        an_count(a, 1);
        if ((st = sums.fetch(s, v)) != HELM_OK) return st;
        est = std::sqrt(v[0]);
        if ((st = an_apply_inv<R>(a, cycles)) != HELM_OK) return st;
        k_an_tfin<R><<<a->nblk, AN_NT, 0, s>>>((const c2*)L0.e, a->U1, L0.typ, n, L0.h, a->alpha, a->k, sums.d);
        an_count(a, 1);
        AN_CK(cudaGetLastError());
        if ((st = sums.fetch(s, v)) != HELM_OK) return st;
        if (!(v[0] > 0.0) || !std::isfinite(v[0])) return HELM_ENONFINITE;
        sc = 1.0 / std::sqrt(v[0]);
        ok = (std::fabs(est - prev) <= tol * est) ? ok + 1 : 0;
        prev = est;
        if (ok >= 2) {
            c1 = true;
            break;
        }
    }
    *smax = est;
    // sigma_min: Lanczos on the real K = A^T D A
    double* buf = nullptr;
    if (cudaMalloc(&buf, 4 * total * sizeof(double)) != cudaSuccess) return HELM_ENOMEM;
    struct Free {
        double* p;
        ~Free() { cudaFree(p); }
    } fr{buf};
    double *vp = buf, *vc = buf + total, *w = buf + 2 * total, *y = buf + 3 * total;
    AN_CK(cudaMemsetAsync(vp, 0, total * sizeof(double), s));
    k_an_lz_scale<<<a->nblk, AN_NT, 0, s>>>(vc, nullptr, 0.0, L0.typ, total, sums.d);
    if ((st = sums.fetch(s, v)) != HELM_OK) return st;
    k_an_lz_scale<<<a->nblk, AN_NT, 0, s>>>(vc, vc, 1.0 / std::sqrt(v[0]), L0.typ, total, sums.d);
    an_count(a, 2);
    const double dp = 1.0 / (a->alpha * a->alpha), de = 1.0 / (a->k * a->k);
    std::vector<double> al, be(1, 0.0);
    double beta = 0.0, theta = 0.0, tprev = 0.0;
    int it2 = 0;
    bool c2ok = false;
    ok = 0;
    for (it2 = 1; it2 <= max_iter; ++it2) {
        k_an_lz_a<<<a->nblk, AN_NT, 0, s>>>(vc, y, L0.typ, n, L0.h, a->sigma, dp, de);
        k_an_lz_at<<<a->nblk, AN_NT, 0, s>>>(y, vc, vp, beta, w, L0.typ, n, L0.h, a->sigma, sums.d);
        an_count(a, 2);
        if ((st = sums.fetch(s, v)) != HELM_OK) return st;
        const double alpha = v[0];
        k_an_lz_orth<<<a->nblk, AN_NT, 0, s>>>(w, vc, alpha, total, sums.d);
        an_count(a, 1);
        AN_CK(cudaGetLastError());
        if ((st = sums.fetch(s, v)) != HELM_OK) return st;
        al.push_back(alpha);
        beta = std::sqrt(v[0]);
        theta = tridiag_max(al, be, (int)al.size());
        be.push_back(beta);
        ok = (std::fabs(theta - tprev) <= tol * theta) ? ok + 1 : 0;
        tprev = theta;
        if (ok >= 2 || !(beta > 1e-300 * theta)) {
            c2ok = true;
            break;
        }
        // v_prev <- v, v <- w / beta (into the old v_prev buffer)
        k_an_lz_scale<<<a->nblk, AN_NT, 0, s>>>(vp, w, 1.0 / beta, L0.typ, total, sums.d);
        an_count(a, 1);
        std::swap(vp, vc);
    }
    AN_CK(cudaStreamSynchronize(s));
    if (!(theta > 0.0) || !std::isfinite(theta)) return HELM_ENONFINITE;
    *smin = 1.0 / std::sqrt(theta);
    *iters = std::max(std::min(it1, max_iter), std::min(it2, max_iter));
    *conv = c1 && c2ok;
    return HELM_OK;
}

}  // namespace

extern "C" {

helm_status helm_annulus_create(helm_annulus** out, int n, double side, double hole, double k, int prec)
{
    if (!out) return HELM_EINVAL;
    *out = nullptr;
    if (n < 16 || n > 16384 || (n & (n - 1))) return HELM_EINVAL;
    if (!(side > 0.0) || !std::isfinite(side) || !(hole > 0.0) || !(hole < 0.5 * side)) return HELM_EINVAL;
    if (!(k >= 0.0) || !std::isfinite(k) || (prec != HELM_PREC_FP64 && prec != HELM_PREC_MIXED)) return HELM_EINVAL;
    helm_annulus* a = new helm_annulus();
    a->N = n;
    a->side = side;
    a->hole = hole;
    a->k = k;
    a->alpha = k * k;
    a->sigma = 0.0;
    a->prec = prec;
    auto fail = [&](helm_status st) { helm_annulus_destroy(a); return st; };
    // a blocking stream: its work is ordered after the caller's work on the legacy default
    // stream (where the inputs were written)
    if (cudaStreamCreate(&a->stream) != cudaSuccess) return fail(HELM_ECUDA);
    if (cudaStreamCreateWithFlags(&a->cap, cudaStreamNonBlocking) != cudaSuccess) return fail(HELM_ECUDA);
    a->ls = a->stream;
    const size_t eb = prec == HELM_PREC_FP64 ? 16 : 8;
    // all levels in one allocation: types, iterate, right-hand side, swept iterate of each
    auto a256 = [](size_t b) { return (b + 255) / 256 * 256; };
    std::vector<std::vector<unsigned char>> types;
    size_t bytes = 0;
    for (int m = n; m >= AN_NC; m /= 2) {
        types.push_back(an_types(m, side, hole));
        if (!an_geometry_ok(types.back(), m)) return fail(HELM_EINVAL);
        const size_t pts = (size_t)(m + 1) * (m + 1);
        bytes += a256(pts) + 3 * a256(pts * eb);
    }
    char* lp = nullptr;
    if (cudaMalloc((void**)&lp, bytes) != cudaSuccess) return fail(HELM_ENOMEM);
    a->allocs.push_back(lp);
    if (cudaMemset(lp, 0, bytes) != cudaSuccess) return fail(HELM_ECUDA);
    for (int m = n; m >= AN_NC; m /= 2) {
        const std::vector<unsigned char>& t = types[a->lev.size()];
        helm_annulus::Level L{};
        L.n = m;
        L.h = side / m;
        const size_t pts = (size_t)(m + 1) * (m + 1);
        const size_t pb = a256(pts * eb);
        L.typ = (unsigned char*)lp;
        L.e = lp + a256(pts);
        L.rhs = (char*)L.e + pb;
        L.e2 = (char*)L.rhs + pb;
        lp += a256(pts) + 3 * pb;
        if (cudaMemcpy(L.typ, t.data(), pts, cudaMemcpyHostToDevice) != cudaSuccess) return fail(HELM_ECUDA);
        // band: the hole's index box [lo, hi]^2 (centred square) widened by AN_BAND nodes
        int lo = m, hi = 0;
        for (int i = 0; i <= m; ++i)
            if (t[(size_t)i * (m + 1) + m / 2] == AN_HOLE) { lo = std::min(lo, i); hi = std::max(hi, i); }
        L.lo = lo;
        L.hi = hi;
        L.b0 = std::max(1, lo - AN_BAND);
        L.b1 = std::min(m - 1, hi + AN_BAND);
        a->lev.push_back(L);
    }
    if (a->lev.size() < 2) return fail(HELM_EINVAL);
    // the coarse tail: levels of at most `top` intervals (at most AN_TAIL_MAX of them)
    const int top = prec == HELM_PREC_FP64 ? AN_TAIL_TOP_D : AN_TAIL_TOP_F;
    for (int l = 0; l < (int)a->lev.size(); ++l)
        if (a->lev[l].n <= top) { a->t0 = l; break; }
    if (a->t0 < 0 || (int)a->lev.size() - a->t0 > AN_TAIL_MAX) return fail(HELM_EUNSUPPORTED);
    {
        const bool d = prec == HELM_PREC_FP64;
        const cudaError_t e = d ? an_attrs<double>() : an_attrs<float>();
        if (e != cudaSuccess) {
            note_error(cudaGetErrorString(e));
            return fail(HELM_ECUDA);
        }
    }
    const long total = (long)(n + 1) * (n + 1);
    a->nblk = grid_for(total);
    void* p = nullptr;
    if (cudaMalloc(&p, total * sizeof(double2) + sizeof(double) * a->nblk + 256) != cudaSuccess)
        return fail(HELM_ENOMEM);
    a->allocs.push_back(p);
    a->U1 = (double2*)p;
    a->part = (double*)((char*)p + total * sizeof(double2));
    a->kmin = (unsigned long long*)((char*)a->part + sizeof(double) * a->nblk);
    a->ctl = (AnCtl*)(a->kmin + 2);
    static_assert(sizeof(AnCtl) + 16 <= 256, "the control follows kmin in the plan's buffer");
    if (cudaMallocHost(&a->h_hist, sizeof(double) * (AN_HIST + 1)) != cudaSuccess) return fail(HELM_ENOMEM);
    helm_status st = helm_annulus_set_shift(a, a->alpha);
    if (st != HELM_OK) return fail(st);
    *out = a;
    return HELM_OK;
}

helm_status helm_annulus_destroy(helm_annulus* a)
{
    if (!a) return HELM_EINVAL;
    if (a->stream) cudaStreamSynchronize(a->stream);
    for (void* p : a->allocs) cudaFree(p);
    if (a->At) cudaFree(a->At);
    an_drop_loop(a);
    if (a->h_hist) cudaFreeHost(a->h_hist);
    if (a->stream) cudaStreamDestroy(a->stream);
    if (a->cap) cudaStreamDestroy(a->cap);
    delete a;
    return HELM_OK;
}

helm_status helm_annulus_set_shift(helm_annulus* a, double alpha)
{
    if (!a || !std::isfinite(alpha) || alpha < a->k * a->k) return HELM_EINVAL;
    an_drop_loop(a);
    a->alpha = alpha;
    a->sigma = (alpha == a->k * a->k) ? 0.0 : alpha - a->k * a->k;
    const auto& C = a->lev.back();
    std::vector<unsigned char> t = an_types(C.n, a->side, a->hole);
    std::vector<double> inv;
    std::vector<int> map;
    if (!an_coarse_inverse(t, C.n, C.h, a->sigma, inv, map)) return HELM_EINVAL;
    if (a->At) cudaFree(a->At);
    a->At = nullptr;
    const int m = (int)map.size();
    a->m = m;
    void* p = nullptr;
    if (cudaMalloc(&p, inv.size() * sizeof(double) + map.size() * sizeof(int)) != cudaSuccess) return HELM_ENOMEM;
    a->At = (double*)p;
    a->map = (int*)(a->At + inv.size());
    std::vector<double> at(inv.size());
    for (int r = 0; r < m; ++r)
        for (int c = 0; c < m; ++c) at[(size_t)c * m + r] = inv[(size_t)r * m + c];
    AN_CK(cudaMemcpy(a->At, at.data(), at.size() * sizeof(double), cudaMemcpyHostToDevice));
    AN_CK(cudaMemcpy(a->map, map.data(), map.size() * sizeof(int), cudaMemcpyHostToDevice));
    int ns[AN_TAIL_MAX];
    const int L = (int)a->lev.size() - a->t0;
    for (int i = 0; i < L; ++i) ns[i] = a->lev[a->t0 + i].n;
    a->tail_bytes = a->prec == HELM_PREC_FP64 ? an_tail_bytes<double>(ns, L, m) : an_tail_bytes<float>(ns, L, m);
    return HELM_OK;
}

helm_status helm_annulus_set_cycle(helm_annulus* a, int nu1, int nu2, int cycles)
{
    if (!a || nu1 < 0 || nu1 > 8 || nu2 < 0 || nu2 > 8 || nu1 + nu2 < 1 || cycles < 1 || cycles > 16)
        return HELM_EINVAL;
    an_drop_loop(a);
    a->nu1 = nu1;
    a->nu2 = nu2;
    a->cycles = cycles;
    return HELM_OK;
}

helm_status helm_annulus_solve(helm_annulus* a, const void* data, void* u, double tol, int max_outer, int* iters,
                               double* res_hist)
{
    if (!a || !(tol >= 0.0) || max_outer < 0) return HELM_EINVAL;
    if (!device_pointer_ok(data) || !device_pointer_ok(u) || data == u) return HELM_EINVAL;
    int status = HELM_MAXITER;
    const helm_status st = (a->prec == HELM_PREC_FP64)
        ? an_solve<double>(a, (const double2*)data, (double2*)u, tol, max_outer, iters, res_hist, &status)
        : an_solve<float>(a, (const double2*)data, (double2*)u, tol, max_outer, iters, res_hist, &status);
    return st != HELM_OK ? st : (helm_status)status;
}

helm_status helm_annulus_exit_times(helm_annulus* a, double c_tau, double tol, int max_outer, void* E_out,
                                    void* L_out, double* kstar)
{
    if (!a || !(c_tau > 0.0) || !std::isfinite(c_tau) || !(tol >= 0.0) || max_outer < 1) return HELM_EINVAL;
    if (!device_pointer_ok(E_out) || !device_pointer_ok(L_out) || E_out == L_out) return HELM_EINVAL;
    // Delta E = -c_tau, dE/dn = 0 and Delta L = 0, dL/dn = 1 (zero on the hole): the outer
    // iteration with k = 0 and no shift, i.e. FP64-refined multigrid solves of A_0
    helm_annulus* z = nullptr;
    helm_status st = helm_annulus_create(&z, a->N, a->side, a->hole, 0.0, a->prec);
    if (st != HELM_OK) return st;
    helm_annulus_set_cycle(z, a->nu1, a->nu2, a->cycles);
    const long total = (long)(a->N + 1) * (a->N + 1);
    std::vector<unsigned char> t = an_types(a->N, a->side, a->hole);
    std::vector<double2> hd(total);
    void* buf = nullptr;
    if (cudaMalloc(&buf, 2 * total * sizeof(double2)) != cudaSuccess) {
        helm_annulus_destroy(z);
        return HELM_ENOMEM;
    }
    double2* dd = (double2*)buf;
    double2* U = dd + total;
    auto done = [&](helm_status s) {
        cudaFree(buf);
        helm_annulus_destroy(z);
        return s;
    };
    for (int which = 0; which < 2; ++which) {
        for (long q = 0; q < total; ++q)
            hd[q] = make_double2(t[q] == AN_PDE ? (which == 0 ? -c_tau : 0.0) : (t[q] == AN_EDGE && which == 1 ? 1.0 : 0.0),
                                 0.0);
        if (cudaMemcpy(dd, hd.data(), total * sizeof(double2), cudaMemcpyHostToDevice) != cudaSuccess)
            return done(HELM_ECUDA);
        int it = 0;
        st = helm_annulus_solve(z, dd, U, tol, max_outer, &it, nullptr);
        if (st != HELM_CONVERGED) return done(st < 0 ? st : HELM_MAXITER);
        k_an_real<<<grid_for(total), AN_NT, 0, z->stream>>>(U, (double*)(which == 0 ? E_out : L_out), total);
        add_launches(1);
    }
    if (kstar) {
        const unsigned long long init = 0x7ff0000000000000ull;      // +inf
        if (cudaMemcpyAsync(z->kmin, &init, sizeof init, cudaMemcpyHostToDevice, z->stream) != cudaSuccess)
            return done(HELM_ECUDA);
        k_an_kstar<<<grid_for(total), AN_NT, 0, z->stream>>>((const double*)E_out, (const double*)L_out,
                                                             z->lev[0].typ, total, z->kmin);
        add_launches(1);
        unsigned long long bits = 0;
        if (cudaMemcpyAsync(&bits, z->kmin, sizeof bits, cudaMemcpyDeviceToHost, z->stream) != cudaSuccess ||
            cudaStreamSynchronize(z->stream) != cudaSuccess)
            return done(HELM_ECUDA);
        double v;
        memcpy(&v, &bits, sizeof v);
        *kstar = v;
    }
    if (cudaStreamSynchronize(z->stream) != cudaSuccess) return done(HELM_ECUDA);
    return done(HELM_OK);
}

helm_status helm_annulus_spectral_radius(helm_annulus* a, int max_iters, double tol, int cycles, double* rho,
                                         double* lambda_re, double* lambda_im, int* iters_done)
{
    if (!a || max_iters < 1 || !(tol > 0.0) || cycles < 1 || cycles > 64) return HELM_EINVAL;
    double r = 0.0, lr = 0.0, li = 0.0;
    int it = 0;
    bool conv = false;
    const helm_status st = (a->prec == HELM_PREC_FP64)
        ? an_spectral<double>(a, max_iters, tol, cycles, &r, &lr, &li, &it, &conv)
        : an_spectral<float>(a, max_iters, tol, cycles, &r, &lr, &li, &it, &conv);
    if (st != HELM_OK) return st;
    if (rho) *rho = r;
    if (lambda_re) *lambda_re = lr;
    if (lambda_im) *lambda_im = li;
    if (iters_done) *iters_done = it;
    return conv ? HELM_OK : HELM_MAXITER;
}

helm_status helm_annulus_condition(helm_annulus* a, int max_iters, double tol, int cycles, double* sigma_max,
                                   double* sigma_min, double* cond, int* iters_done)
{
    if (!a || max_iters < 1 || !(tol > 0.0) || cycles < 1 || cycles > 64 || !(a->k > 0.0)) return HELM_EINVAL;
    double smax = 0.0, smin = 0.0;
    int it = 0;
    bool conv = false;
    const helm_status st = (a->prec == HELM_PREC_FP64)
        ? an_singular<double>(a, max_iters, tol, cycles, &smax, &smin, &it, &conv)
        : an_singular<float>(a, max_iters, tol, cycles, &smax, &smin, &it, &conv);
    if (st != HELM_OK) return st;
    if (sigma_max) *sigma_max = smax;
    if (sigma_min) *sigma_min = smin;
    if (cond) *cond = smax / smin;
    if (iters_done) *iters_done = it;
    return conv ? HELM_OK : HELM_MAXITER;
}

}  // extern "C"
