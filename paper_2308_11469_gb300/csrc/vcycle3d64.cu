// 3D multigrid level kernels in FP64.
//
// Operations, colours and weights are those of the generic kernels (vcycle.cu); what differs
// is what bounds them.  An SM serves about 2 FP64 lanes a clock (a warp's FP64 instruction
// holds its sub-core's pipe for 64 clocks) beside 64 integer lanes, so these kernels
//  * number their nodes over all lanes of small blocks (a warp per row of 15 nodes leaves half
//    of the lanes idle and a few SMs at work),
//  * let part of the warps form their sums in 64-bit fixed point on the values' own scale
//    (fixed_win.cuh: exact sums, one rounding), so that both pipes work,
//  * add only the distinct corners of an interpolated node (an even index has one per axis).
#include "launch.h"
#include "pdl.cuh"
#include "fixed_win.cuh"

namespace helm {
namespace {

constexpr int K3_NT = 128;

struct Lev3 {
    int n, pitch;
    long P, PL;                 // row and plane strides
    __device__ explicit Lev3(const LevelDesc& L) : n(L.n), pitch(L.pitch), P(L.pitch), PL((long)L.pitch * L.rows) {}
    __device__ long row(int y, int z) const { return z * PL + y * P; }
    __device__ int x(int i) const { return xslot<3>(i, pitch); }
};

// Of K3_DEN consecutive warps, those that sum in fixed point (half-sweeps: 7 FP64 operations a
// component against about 150 integer ones; restrictions: 28 against 500).  127^3 solve, V(0,2),
// with 1, 2, 3 and 4 of 4: 7.63, 7.04, 6.76 and 6.99 ms (11.1 with the generic kernels); a
// half-sweep of level 127 29 us against 37, the restriction 27 against 40, the prolongation 28
// against 46, the levels below 31 5-7 us a launch against 8-19.
constexpr int K3_DEN = 4, K3_SWEEP = 3, K3_RESTRICT = 3;
__device__ __forceinline__ bool k3_fixed(int t, int num) { return (t >> 5) % K3_DEN < num; }

// One red-black half-sweep; modes as k_rbgs
__global__ void __launch_bounds__(K3_NT)
k_rbgs64(const InstDesc* __restrict__ insts, const InstState* __restrict__ st, const MgItem* __restrict__ items,
         int color, int mode)
{
    pdl_wait();
    pdl_trigger();
    const MgItem item = items[blockIdx.y];
    const InstState sv = st[item.inst];
    if (sv.status != HELM_ST_ACTIVE) return;
    const LevelDesc L = insts[item.inst].lev[item.level];
    const Lev3 G(L);
    const int n = G.n, half = (n + 1) >> 1, total = n * n * half;
    double2* __restrict__ e = (double2*)L.e;
    const double2* __restrict__ r = (const double2*)lev_rhs(L, item.level, sv.it);
    const FxH2 hh(L.h2);
    const double inv = L.dinv;                     // 1 / (6 + sigma h^2)
    const bool zi = (mode == 2) || (mode == 1 && item.level > 0);
    for (int t = blockIdx.x * K3_NT + threadIdx.x; t < total; t += gridDim.x * K3_NT) {
        const int row = t / half, j = t - row * half;
        const int y = row % n + 1, z = row / n + 1;
        const int xa = 2 * j + 1;                  // pair {xa, xa + 1}
        const bool first = ((xa + y + z) & 1) == color;
        const int xc = first ? xa : xa + 1, xo = first ? xa + 1 : xa;
        const long rb = G.row(y, z);
        if (xc <= n) {
            const long o = rb + G.x(xc);
            const double2 rr = r[o];
            double2 v;
            if (zi) {                              // all neighbours are zero
                v.x = -hh.h2 * rr.x * inv;
                v.y = -hh.h2 * rr.y * inv;
            } else {
                const double2 a = e[rb + G.x(xc - 1)], b = e[rb + G.x(xc + 1)];
                const double2 c = e[o - G.P], d = e[o + G.P], f = e[o - G.PL], g = e[o + G.PL];
                const int er = fx_exp2(rr);
                const int em = max(max(max(fx_exp2(a), fx_exp2(b)), max(fx_exp2(c), fx_exp2(d))),
                                   max(max(fx_exp2(f), fx_exp2(g)), er ? er + hh.add : 0));
                if (k3_fixed(t, K3_SWEEP) && hh.usable(em)) {
                    const longlong2 A = fx_q2(a, em), B = fx_q2(b, em), C = fx_q2(c, em), D = fx_q2(d, em);
                    const longlong2 F = fx_q2(f, em), H = fx_q2(g, em), Q = hh.q2(rr, em);
                    const double2 s = fx_d2(make_longlong2(((A.x + B.x) + (C.x + D.x)) + ((F.x + H.x) - Q.x),
                                                           ((A.y + B.y) + (C.y + D.y)) + ((F.y + H.y) - Q.y)), em);
                    v = make_double2(s.x * inv, s.y * inv);
                } else {
                    double sx = a.x + b.x + c.x + d.x, sy = a.y + b.y + c.y + d.y;
                    sx += f.x + g.x;
                    sy += f.y + g.y;
                    v.x = (sx - hh.h2 * rr.x) * inv;
                    v.y = (sy - hh.h2 * rr.y) * inv;
                }
            }
            e[o] = v;
        }
        if (zi && xo <= n) e[rb + G.x(xo)] = make_double2(0.0, 0.0);
    }
}

// Residual and full weighting; modes as k_restrict
__global__ void __launch_bounds__(K3_NT)
k_restrict64(const InstDesc* __restrict__ insts, const InstState* __restrict__ st, const MgItem* __restrict__ items,
             int mode)
{
    pdl_wait();
    pdl_trigger();
    const MgItem item = items[blockIdx.y];
    const InstState sv = st[item.inst];
    if (sv.status != HELM_ST_ACTIVE) return;
    const LevelDesc Fd = insts[item.inst].lev[item.level];
    const LevelDesc Cd = insts[item.inst].lev[item.level + 1];
    const Lev3 F(Fd), C(Cd);
    const int nc = C.n, total = nc * nc * nc;
    const double2* __restrict__ e = (const double2*)Fd.e;
    const double2* __restrict__ r = (const double2*)lev_rhs(Fd, item.level, sv.it);
    double2* __restrict__ cr = (double2*)Cd.rhs;
    double2* __restrict__ ce = (double2*)Cd.e;
    const bool ez = (mode == 2) || (mode == 1 && item.level > 0);
    const double sig = insts[item.inst].sigma;
    const double ih2 = ez ? 0.0 : 1.0 / Fd.h2;     // (a division costs a warp 1300 clocks)
    for (int t = blockIdx.x * K3_NT + threadIdx.x; t < total; t += gridDim.x * K3_NT) {
        const int row = t / nc, X = t - row * nc + 1, Y = row % nc + 1, Z = row / nc + 1;
        const long oc = C.row(Y, Z) + C.x(X);
        const int x0 = F.x(2 * X - 1), x1 = F.x(2 * X), x2 = F.x(2 * X + 1);
        double ax = 0.0, ay = 0.0;
        if (ez) {
            if (k3_fixed(t, K3_RESTRICT)) {
                int ex = 0;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const double2* p = r + F.row(2 * Y + k % 3 - 1, 2 * Z + k / 3 - 1);
                    ex = max(ex, max(max(fx_exp2(p[x0]), fx_exp2(p[x2])), fx_exp2(p[x1])));
                }
                // 64 times the largest value at most: 4 bits of the scale for the sum
                ex += 4;
                if (fx_usable(ex)) {
                    longlong2 s = make_longlong2(0, 0);
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        const double2* p = r + F.row(2 * Y + k % 3 - 1, 2 * Z + k / 3 - 1);
                        const longlong2 a = fx_q2(p[x0], ex), m = fx_q2(p[x1], ex), b = fx_q2(p[x2], ex);
                        const int w = (k % 3 == 1) + (k / 3 == 1);
                        s.x += ((a.x + b.x) + 2 * m.x) << w;
                        s.y += ((a.y + b.y) + 2 * m.y) << w;
                    }
                    cr[oc] = fx_d2(s, ex - 6);
                    continue;
                }
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const double2* p = r + F.row(2 * Y + k % 3 - 1, 2 * Z + k / 3 - 1);
                const double w = (k % 3 == 1 ? 2.0 : 1.0) * (k / 3 == 1 ? 2.0 : 1.0);
                const double2 a = p[x0], m = p[x1], b = p[x2];
                ax += w * a.x;
                ay += w * a.y;
                ax += 2.0 * w * m.x;
                ay += 2.0 * w * m.y;
                ax += w * b.x;
                ay += w * b.y;
            }
            cr[oc] = make_double2(ax * (1.0 / 64.0), ay * (1.0 / 64.0));
            continue;
        }
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy) {
                const long rb = F.row(2 * Y + dy, 2 * Z + dz);
                const double wr = (dz == 0 ? 2.0 : 1.0) * (dy == 0 ? 2.0 : 1.0);
                for (int dx = -1; dx <= 1; ++dx) {
                    const double w = wr * (dx == 0 ? 2.0 : 1.0);
                    const int x = 2 * X + dx;
                    const long o = rb + F.x(x);
                    const double2 c = e[o], a = e[rb + F.x(x - 1)], b = e[rb + F.x(x + 1)];
                    const double2 u = e[o - F.P], d = e[o + F.P], f = e[o - F.PL], g = e[o + F.PL];
                    double sx = a.x + b.x + u.x + d.x, sy = a.y + b.y + u.y + d.y;
                    sx += f.x + g.x;
                    sy += f.y + g.y;
                    const double2 rr = r[o];
                    ax += w * ((rr.x - (sx - 6.0 * c.x) * ih2) + sig * c.x);
                    ay += w * ((rr.y - (sy - 6.0 * c.y) * ih2) + sig * c.y);
                }
            }
        cr[oc] = make_double2(ax * (1.0 / 64.0), ay * (1.0 / 64.0));
        ce[oc] = make_double2(0.0, 0.0);
    }
}

// Trilinear prolongation and correction; modes and skip0 as k_prolong.  A thread owns the fine
// pair 2 p + 1, 2 p + 2 of a row; with skip0 one node of it.
__global__ void __launch_bounds__(K3_NT)
k_prolong64(const InstDesc* __restrict__ insts, const InstState* __restrict__ st, const MgItem* __restrict__ items,
            int mode, int skip0)
{
    pdl_wait();
    pdl_trigger();
    const MgItem item = items[blockIdx.y];
    if (st[item.inst].status != HELM_ST_ACTIVE) return;
    const LevelDesc Fd = insts[item.inst].lev[item.level];
    const LevelDesc Cd = insts[item.inst].lev[item.level + 1];
    const Lev3 F(Fd), C(Cd);
    const int n = F.n, half = (n + 1) >> 1, total = n * n * half;
    double2* __restrict__ e = (double2*)Fd.e;
    const double2* __restrict__ ce = (const double2*)Cd.e;
    const bool ez = (mode == 2) || (mode == 1 && item.level > 0);
    for (int t = blockIdx.x * K3_NT + threadIdx.x; t < total; t += gridDim.x * K3_NT) {
        const int row = t / half, p = t - row * half;
        const int y = row % n + 1, z = row / n + 1;
        const long rb = F.row(y, z);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int x = 2 * p + 1 + k;
            if (x > n || (skip0 && ((x + y + z) & 1) == 0)) continue;
            // the corner rows (one or two an axis), of each the column x / 2 or two
            double sx = 0.0, sy = 0.0, w = 1.0;
            const int X = C.x(x >> 1), X1 = C.x((x >> 1) + 1);
            auto add = [&](int yy, int zz, bool start) {
                const double2* q = ce + C.row(yy, zz);
                double2 v = q[X];
                if (x & 1) {
                    const double2 u = q[X1];
                    v.x += u.x;
                    v.y += u.y;
                }
                if (start) {
                    sx = v.x;
                    sy = v.y;
                } else {
                    sx += v.x;
                    sy += v.y;
                }
            };
            const int y0 = y >> 1, z0 = z >> 1;
            add(y0, z0, true);
            if (y & 1) add(y0 + 1, z0, false);
            if (z & 1) {
                add(y0, z0 + 1, false);
                if (y & 1) add(y0 + 1, z0 + 1, false);
            }
            if (x & 1) w = 0.5;
            if (y & 1) w *= 0.5;
            if (z & 1) w *= 0.5;
            const long o = rb + F.x(x);
            double2 v = make_double2(w * sx, w * sy);
            if (!ez) {
                const double2 c = e[o];
                v = make_double2(fma(w, sx, c.x), fma(w, sy, c.y));
            }
            e[o] = v;
        }
    }
}

dim3 grid64(int work, int nitems)
{
    const int b = (work + K3_NT - 1) / K3_NT;
    return dim3(b < 1 ? 1 : (b > 152 * 64 ? 152 * 64 : b), nitems);
}

}  // namespace

cudaError_t launch_rbgs64(const InstDesc* insts, const InstState* st, const MgItem* items, int nitems, int work,
                          int color, int mode, cudaStream_t s)
{
    launch_k(k_rbgs64, grid64(work, nitems), dim3(K3_NT), 0, s, insts, st, items, color, mode);
    return cudaGetLastError();
}

cudaError_t launch_restrict64(const InstDesc* insts, const InstState* st, const MgItem* items, int nitems, int work,
                              cudaStream_t s, int mode)
{
    launch_k(k_restrict64, grid64(work, nitems), dim3(K3_NT), 0, s, insts, st, items, mode);
    return cudaGetLastError();
}

cudaError_t launch_prolong64(const InstDesc* insts, const InstState* st, const MgItem* items, int nitems, int work,
                             cudaStream_t s, int mode, int skip0)
{
    launch_k(k_prolong64, grid64(work / 2, nitems), dim3(K3_NT), 0, s, insts, st, items, mode, skip0);
    return cudaGetLastError();
}

cudaError_t setup_3d64()
{
    cudaError_t e;
    if ((e = max_carveout(k_rbgs64)) != cudaSuccess) return e;
    if ((e = max_carveout(k_restrict64)) != cudaSuccess) return e;
    return max_carveout(k_prolong64);
}

}  // namespace helm
