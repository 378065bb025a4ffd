// Pieces of the outer (FP64) iteration that its kernels share (outer.cu, small2d.cu): the
// status rule, fixed-order reductions, the step control and the per-node residual.
#pragma once
#include <type_traits>

#include "launch.h"
#include "float_sum.cuh"
#include "fixed_lap.cuh"
#include "fixed_win.cuh"

namespace helm {
namespace {

constexpr int NTH = 256;

// FP64 -> inner precision and back; for complex64 the format changes run on the
// integer pipes (fp_bits.cuh), leaving the FP64 pipe to the update and the stencil.
__device__ __forceinline__ float2 to_inner_f(double2 v) { return make_float2(d2f_bits(v.x), d2f_bits(v.y)); }
template <typename R> struct Inner;
template <> struct Inner<float> {
    static __device__ __forceinline__ float2 from(double2 v) { return to_inner_f(v); }
    static __device__ __forceinline__ double widen(float x) { return f2d_bits(x); }
};
template <> struct Inner<double> {
    static __device__ __forceinline__ double2 from(double2 v) { return v; }
    static __device__ __forceinline__ double widen(double x) { return x; }
};

// Status rule (the paper only reports "converges" / "diverges"; this project's reading):
// CONVERGED when relres <= tol; DIVERGED when relres > 1e4, or when N >= 20, relres has
// not decreased for 10 consecutive steps and has grown to at least twice its smallest
// value so far (stagnation at the rounding floor is not divergence); NONFINITE on NaN /
// Inf; MAXITER at max_outer.
// relres_N = ||r_N|| / ||b||, b the lifted right-hand side (f minus the wall values'
// contribution to the stencil): with the paper's zero start r_0 = b and relres_0 = 1; a
// starting iterate that already solves the system well starts with a small relres.
// mode 0: `second` is ||b||^2 (mode 1: not used; instance_last records the increment's norm).
// The outcome after step N (0: the start) with relative residual rel, into s (run, rmin,
// prev, status).
__device__ __forceinline__ void status_rule(const InstDesc& I, InstState& s, double rel, int N, bool zero)
{
    int out = HELM_ST_ACTIVE;
    if (!isfinite(rel)) out = -4;                                   // HELM_ENONFINITE
    else if (rel <= I.tol || zero) out = 0;                         // CONVERGED
    else if (rel > 1e4) out = 2;                                    // DIVERGED
    else {
        if (N != 0) s.run = (rel >= s.prev) ? s.run + 1 : 0;
        s.rmin = fmin(s.rmin, rel);
        if (N >= 20 && s.run >= 10 && rel >= 2.0 * s.rmin) out = 2; // DIVERGED
        else if (N >= I.max_outer) out = 1;                         // MAXITER
    }
    s.prev = rel;
    s.status = out;
}

__device__ void finalize(const InstDesc& I, InstState* stp, double norm2, double second, int mode)
{
    InstState s = *stp;
    const double norm = sqrt(norm2);
    double rel;
    int N;
    if (mode == 0) {
        N = 0;
        const double nb = sqrt(second);
        s.norm0 = (nb > 0.0) ? nb : norm;      // zero data: measure against r_0 itself
        s.run = 0;
        rel = (norm == 0.0) ? 0.0 : norm / s.norm0;
        if (!isfinite(norm) || !isfinite(nb)) rel = norm + nb;
        s.rmin = rel;
    } else {
        s.it += 1;
        N = s.it;
        rel = norm / s.norm0;
    }
    I.hist[N] = rel;
    status_rule(I, s, rel, N, mode == 0 && norm == 0.0);
    *stp = s;
}

// Block-wide sums / maxima in a fixed order (xor-shuffle in T, then the warps' values in
// order, in FP64).  `sum2`: the second channel is summed (mode 0, ||b||^2) instead of
// maximised (max |e|^2, non-negative: FP64 maxima are taken on the bits).  Mode 1 reduces its
// complex64-derived values in FP32 within a warp, keeping the shuffle tree off the FP64 pipe, and
// adds the warps' sums to FP64's accuracy (float_sum.cuh); the result (thread 0) is FP64 either
// way.  live: only the first `live` warps hold values.
template <typename T>
__device__ __forceinline__ void block_reduce(T a, T m, double& ra, double& rm, double* sa, double* sm,
                                             bool sum2, int live = 32)
{
    const int nw = min((int)(blockDim.x >> 5), live), w = threadIdx.x >> 5;
    if constexpr (std::is_same<T, float>::value) {
        float* const fa = reinterpret_cast<float*>(sa);
        float* const fm = reinterpret_cast<float*>(sm);
        if (w < nw) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                const float mo = __shfl_xor_sync(0xffffffffu, m, o);
                m = m > mo ? m : mo;
            }
            if ((threadIdx.x & 31) == 0) {
                fa[w] = a;
                fm[w] = m;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float mf = 0.f;
            for (int i = 0; i < nw; ++i) mf = fmaxf(mf, fm[i]);
            ra = sum_floats(fa, nw);
            rm = widen_any(mf);
        }
    } else {
        if (w < nw) {
            long long mi = __double_as_longlong(m);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                if (sum2) m += __shfl_xor_sync(0xffffffffu, m, o);
                else mi = max(mi, __shfl_xor_sync(0xffffffffu, mi, o));
            }
            if ((threadIdx.x & 31) == 0) {
                sa[w] = a;
                sm[w] = sum2 ? m : __longlong_as_double(mi);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            ra = sa[0];
            rm = sm[0];
            for (int i = 1; i < nw; ++i) {
                ra += sa[i];
                rm = sum2 ? rm + sm[i]
                          : __longlong_as_double(max(__double_as_longlong(rm), __double_as_longlong(sm[i])));
            }
        }
    }
}

// End of an outer step, run by one whole CTA once every instance's status is final: is
// any instance still iterating?  Counts the step, applies the step budget of this launch
// and sets the loop condition of the graph's WHILE node.
__device__ void step_end(const InstState* st, int nscan, int* ctrl, int use_cond,
                         unsigned long long cond_handle)
{
    __shared__ int any_active;
    if (threadIdx.x == 0) any_active = 0;
    __syncthreads();
    int a = 0;
    for (int i = threadIdx.x; i < nscan; i += blockDim.x)
        a |= (__ldcg(&st[i].status) == HELM_ST_ACTIVE);
    if (a) atomicOr(&any_active, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int go = any_active;
        const int done = ctrl[0] + 1;
        ctrl[0] = done;
        if (done >= ctrl[1]) go = 0;          // step budget of this launch
        ctrl[2] = go;
        if (use_cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond_handle, go ? 1u : 0u);
    }
}

// Step control folded into the residual launch (ctrl == nullptr: not folded).  Every
// instance of the launch arrives once -- an iterating instance from the CTA that
// finalised its status, a finished one from the CTA of its first tile -- and the last
// arrival (launch-wide ticket ctrl[3]) ends the step.
struct StepCtl {
    int* ctrl;
    int nscan;                  // status entries to scan (descriptor slots)
    int ninst;                  // instances with tiles in this launch
    int use_cond;
    unsigned long long cond;
};

__device__ void step_arrive(const InstState* st, const StepCtl& c)
{
    __shared__ int last_arrival;
    if (threadIdx.x == 0) {
        __threadfence();                      // this instance's status before the ticket
        last_arrival = (atomicAdd(&c.ctrl[3], 1) == c.ninst - 1);
    }
    __syncthreads();
    if (!last_arrival) return;
    __threadfence();
    step_end(st, c.nscan, c.ctrl, c.use_cond, c.cond);
    if (threadIdx.x == 0) c.ctrl[3] = 0;
}

// The CTA that wrote an instance's last partial: sum the nb partials in tile order,
// apply the status rule, and (folded step control) arrive for the step.  The partials are
// read by the first NTH threads whatever the block size (threads beyond add zeros, which
// leaves sums and maxima of non-negative values unchanged), so a launch with larger CTAs
// reduces in the same order as the residual kernels.
// sa, sm: shared scratch of one double per warp of the CTA.
__device__ void instance_last(const InstDesc& I, InstState* stp, int mode, const InstState* st_all,
                              const StepCtl& c, double* sa, double* sm)
{
    const int nb = I.nres_blocks;
    __threadfence();
    double ta = 0.0, tm = 0.0;
    long long ti = 0;
    if ((int)threadIdx.x < NTH)
        for (int b = threadIdx.x; b < nb; b += NTH) {
            ta += __ldcg(I.part + b);
            const double x = __ldcg(I.part + nb + b);
            if (mode == 0) tm += x;
            else ti = max(ti, __double_as_longlong(x));
        }
    if (mode != 0) tm = __longlong_as_double(ti);
    const int it = stp->it;
    __syncthreads();
    double fa = 0.0, fm = 0.0;
    block_reduce<double>(ta, tm, fa, fm, sa, sm, mode == 0, (min(nb, NTH) + 31) >> 5);
    if (threadIdx.x == 0) sm[0] = fm;
    __syncthreads();
    // the increment's norm by another warp, beside relres
    if (mode != 0 && threadIdx.x == 32) I.einf[it] = sqrt(sm[0]);
    if (threadIdx.x == 0) {
        finalize(I, stp, fa, fm, mode);
        *I.count = 0u;
    }
    if (c.ctrl) step_arrive(st_all, c);
}

// Write this tile's partials; the last tile of the instance reduces them all.
template <typename T>
__device__ void tile_done(const InstDesc& I, InstState* stp, int tile, T ta0, T tm0, int mode,
                          const InstState* st_all, const StepCtl& c)
{
    __shared__ double sa[NTH / 32], sm[NTH / 32];
    __shared__ int last;
    double a = 0.0, m = 0.0;
    block_reduce<T>(ta0, tm0, a, m, sa, sm, mode == 0);
    if (threadIdx.x == 0) {
        I.part[tile] = a;
        I.part[I.nres_blocks + tile] = m;
        __threadfence();
        const unsigned prev = atomicAdd(I.count, 1u);
        last = (prev == (unsigned)(I.nres_blocks - 1));
    }
    __syncthreads();
    if (!last) return;
    instance_last(I, stp, mode, st_all, c, sa, sm);
}

// r = f - (Delta_h + k^2 + i p) u at one node: f - k^2 u - (numerator) / h^2, the
// Laplacian numerator (sum of the neighbours - 2D u) summed exactly in fixed point
// (fixed_lap.cuh) on the scale emax, u in FP64, and for DAMP the coupling - i p u.
// helm_resid2d_fx: FC, FA, FB, FD, FU are the fixed-point images of the 2D node and its
// four neighbours (a, b west / east, d, u south / north).
template <bool DAMP>
__device__ __forceinline__ double2 helm_resid_fx(double2 c, long long lx, long long ly, double2 fv, double mih2,
                                                 double mk2, double damp, int emax)
{
    double2 r;
    r.x = fma(fx_to_double(lx, emax), mih2, fma(c.x, mk2, fv.x));
    r.y = fma(fx_to_double(ly, emax), mih2, fma(c.y, mk2, fv.y));
    if constexpr (DAMP) {
        r.x = fma(c.y, damp, r.x);
        r.y = fma(c.x, -damp, r.y);
    }
    return r;
}

template <bool DAMP>
__device__ __forceinline__ double2 helm_resid2d_fx(double2 c, longlong2 FC, longlong2 FA, longlong2 FB,
                                                   longlong2 FD, longlong2 FU, double2 fv, double mih2,
                                                   double mk2, double damp, int emax)
{
    const long long lx = ((FA.x + FB.x) + (FD.x + FU.x)) - 4 * FC.x;
    const long long ly = ((FA.y + FB.y) + (FD.y + FU.y)) - 4 * FC.y;
    return helm_resid_fx<DAMP>(c, lx, ly, fv, mih2, mk2, damp, emax);
}

// helm_resid2d_fx with f - k^2 u already formed (g)
template <bool DAMP>
__device__ __forceinline__ double2 helm_resid2d_g(double2 c, longlong2 FC, longlong2 FA, longlong2 FB, longlong2 FD,
                                                  longlong2 FU, double2 g, double mih2, double damp, int emax)
{
    const long long lx = ((FA.x + FB.x) + (FD.x + FU.x)) - 4 * FC.x;
    const long long ly = ((FA.y + FB.y) + (FD.y + FU.y)) - 4 * FC.y;
    double2 r = make_double2(fma(fx_to_double(lx, emax), mih2, g.x), fma(fx_to_double(ly, emax), mih2, g.y));
    if constexpr (DAMP) {
        r.x = fma(c.y, damp, r.x);
        r.y = fma(c.x, -damp, r.y);
    }
    return r;
}

// scale exponent of a window from its largest biased exponent (see fixed_lap.cuh); -1:
// no fixed-point scale (a value above 2^1007, an infinity or a NaN)
__device__ __forceinline__ int fx_scale(int emax_raw)
{
    return emax_raw > FX_EMAX ? -1 : max(emax_raw, FX_EMIN);
}

__device__ __forceinline__ longlong2 fx_fix2(double2 v, int emax)
{
    return make_longlong2(fx_fix(v.x, emax), fx_fix(v.y, emax));
}

// The residual window of a tile is its (TX + 2) x (TY + 2) nodes; its 1-node ring has
// 2 (TX + 2) + 2 TY nodes, numbered: top row, bottom row, left column, right column.
template <int TX, int TY>
__device__ __forceinline__ void ring_node(int t, int& lx, int& ly)
{
    if (t < TX + 2) { lx = t; ly = 0; }
    else if (t < 2 * (TX + 2)) { lx = t - (TX + 2); ly = TY + 1; }
    else if (t < 2 * (TX + 2) + TY) { lx = 0; ly = t - 2 * (TX + 2) + 1; }
    else { lx = TX + 1; ly = t - 2 * (TX + 2) - TY + 1; }
}

// |v|^2 of an inner-precision complex value, rounded the same way in every kernel
template <typename C>
__device__ __forceinline__ auto abs2(C v) -> decltype(v.x) { return fma(v.y, v.y, v.x * v.x); }

}  // namespace
}  // namespace helm
