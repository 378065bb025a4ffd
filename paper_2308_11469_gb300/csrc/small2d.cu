// Whole solves of small 2D grids (complex64 cycles, n = 31 or 63) in one launch.
//
// One outer step of such a grid is a few microseconds of work, but as separate launches it
// took a one-CTA cycle and a four-CTA residual: 17.4 + 19.9 us at 63^2, launch and memory
// latency almost throughout.  Here a thread-block cluster of CS CTAs keeps a solve on chip
// for all the steps of a call: u and f of a band of rows in each CTA's registers, the levels
// in its shared memory.
//
//  * The V-cycle runs in every CTA on the same right-hand side (the one-CTA tail's code, so
//    the same bits): its phases are bound by latency, and sharing them out would put a
//    cluster barrier behind every half-sweep.  No correction has to be exchanged.
//  * The FP64 part is bound by the FP64 rate of an SM (6 operations a node at 2 a clock:
//    5.8 us on one SM at 63^2), so it is shared out: CTA c updates and differences the
//    rows of its band (and updates the row on either side, which its stencil reads).
//  * Two cluster barriers a step: behind the tiles' largest exponents (the fixed-point
//    scale of a 32 x 32 residual tile is that of its whole window, as in k_residual2d, so
//    residuals are the same whatever CS is) and behind the bands' new residuals, which go
//    straight into the right-hand sides of all CTAs (their cycles are over by then).
//  * Norms are formed by every CTA in k_residual2d's order; all CTAs reach the same outcome.
//    A warp's FP64 instruction holds its sub-core's pipe for 64 clocks however few lanes it
//    serves, so a step compares squared norms as integers and leaves the roots and quotients
//    of relres to the steps that need them: many steps' at once, a lane each (5.5 K -> 1.2 K
//    clocks a step).
//
// Iterates, residuals and histories are those of the launch-by-launch path bit for bit.
// 63^2 plane-wave cavity, V(2,2), 12 steps: 317 us a solve against 501 us (a step 18 us, its
// V-cycle 11.5); 275 with one round trip to the host a solve.
#include <atomic>

#include <cooperative_groups.h>

#include "launch.h"
#include "pdl.cuh"
#include "resid.cuh"
#include "tail_levels.cuh"

namespace helm {
namespace {

namespace cg = cooperative_groups;

template <int N0, int CS> struct SmallLay {
    static constexpr int S = N0 + 2;
    static constexpr int RB = (N0 + 1) / CS;             // rows of a band (the last one: one fewer)
    static constexpr int WN = (RB + 2) * S;              // its window of u: one row more on either side
    static constexpr int NPT = (WN + TNT - 1) / TNT;     // window nodes of a thread
    static constexpr int TX = (N0 + 31) / 32;            // residual tiles per axis
    static constexpr size_t LEVELS = (tail_bytes<2, float, N0>() + 15) & ~(size_t)15;
    static constexpr size_t U_BYTES = (size_t)WN * sizeof(double2);
    static constexpr size_t BYTES = LEVELS + U_BYTES;
    static_assert(BYTES <= 227 * 1024 - 1024, "shared memory of one CTA");
};

template <int N0, int CS, bool DAMP>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(TNT, 1)
k_small2d(const InstDesc* __restrict__ insts, InstState* __restrict__ st, const MgItem* __restrict__ items,
          int nu1, int nu2, int cycles, const float* __restrict__ xtab, StepCtl ctl)
{
    typedef SmallLay<N0, CS> Y;
    constexpr int S = Y::S, RB = Y::RB, NPT = Y::NPT, TX = Y::TX, NT = TX * TX;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* const base = reinterpret_cast<float2*>(smem_raw);
    float* const xscr = reinterpret_cast<float*>(base + tail_elems<2, N0>());
    double2* const U = reinterpret_cast<double2*>(smem_raw + Y::LEVELS);
    __shared__ int own_ex[NT], all_ex[2][NT];             // this band's / the cluster's exponents
    __shared__ float sa[8 * NT], sm[8 * NT];              // per warp: sum |r|^2, max |e|^2
    __shared__ double pend_n[32], pend_m[32];             // the steps whose relres is still to be formed
    __shared__ InstState sst;
    __shared__ int s_budget, s_last;
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cl.block_rank();
    // host-written tables before the wait; the descriptor of a plan's solve is not: k_begin wrote it
    if constexpr (tail_exact<2, float, N0>())
        for (int i = tid; i < XTAB_FLOATS; i += TNT) xscr[i] = xtab[i];
    pdl_wait();
    pdl_trigger();
    const MgItem item = items[blockIdx.x / CS];
    const InstDesc& I = insts[item.inst];
    const LevelDesc L0 = I.lev[0];
    const float sigma = I.sigf;
    if (tid == 0) {
        sst = st[item.inst];
        // steps this launch may make (written by the launch's last arrival only, which every
        // CTA's read precedes)
        s_budget = ctl.ctrl[1] - __ldcg(&ctl.ctrl[0]);
    }
    if (tid < 2 * NT) (&all_ex[0][0])[tid] = 0;
    __syncthreads();
    const int it0 = sst.it;
    const int budget = s_budget;
    int done = 0;
    if (sst.status == HELM_ST_ACTIVE && budget > 0) {
        float2* const E = base;
        float2* const Rr = base + Lv<2, N0>::SZ;
        const float2* __restrict__ gr = (const float2*)lev_rhs(L0, 0, it0);
        const double2* __restrict__ uin = I.u[it0 & 1];
        const double2* __restrict__ f = I.f;
        const int row0 = 1 + rank * RB;                   // first row of the band
        double2 u[NPT], fv[NPT];
#pragma unroll
        for (int j = 0; j < NPT; ++j) {
            const int q = tid + j * TNT, wy = q / S, gx = q - wy * S, gy = row0 - 1 + wy;
            u[j] = make_double2(0.0, 0.0);
            fv[j] = u[j];
            if (q < Y::WN && gy <= N0 + 1) {
                u[j] = uin[gy * S + gx];
                if (wy >= 1 && wy <= RB && gy <= N0 && gx >= 1 && gx <= N0)
                    fv[j] = f[(size_t)(gy - 1) * N0 + (gx - 1)];
            }
        }
        for (int q = tid; q < S * S; q += TNT) {
            const int y = q / S, x = q - y * S;
            const bool in = y >= 1 && y <= N0 && x >= 1 && x <= N0;
            Rr[y * S + ix<N0>(x)] = in ? gr[(size_t)y * L0.pitch + x] : make_float2(0.f, 0.f);
        }
        const double mih2 = -I.ih2, mk2 = -I.k2, damp = I.damp;
        // squared norm (as an ordered integer) at which relres reaches tol, a few ulps above;
        // the last step's squared norm (none yet: the first step forms its relres at once)
        const double tn = I.tol * sst.norm0;
        const long long conv2 = __double_as_longlong(tn * tn) + 64;
        long long prev2 = 0;
        int npend = 0;                                    // (warp 0's)
        cl.sync();                                        // every CTA of the cluster is set up
        int par = 0;
        for (;;) {
            for (int c = 0; c < cycles; ++c) {
                // the iterates start from zero: all levels', or the coarse ones' (a level that
                // is solved exactly is overwritten)
                if (c == 0) t_clear<2, float, N0>(base);
                __syncthreads();
                t_vcycle<2, float, N0, TNT / 32>(base, L0.hf, sigma, &I.lev[0], nu1, nu2, xscr, c == 0);
            }
            // u_{N+1} = u_N + e_N on the band's window, and its largest exponents per tile
            if (tid < NT) {
                own_ex[tid] = 0;
                all_ex[par ^ 1][tid] = 0;                 // read a step ago, raised again a step on
            }
            __syncthreads();
            int ex[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) ex[t] = 0;
#pragma unroll
            for (int j = 0; j < NPT; ++j) {
                const int q = tid + j * TNT, wy = q / S, gx = q - wy * S, gy = row0 - 1 + wy;
                if (q >= Y::WN || gy > N0 + 1) continue;
                if (gy >= 1 && gy <= N0 && gx >= 1 && gx <= N0) {
                    const float2 ev = E[gy * S + ix<N0>(gx)];
                    u[j].x += Inner<float>::widen(ev.x);
                    u[j].y += Inner<float>::widen(ev.y);
                }
                U[q] = u[j];
                const int e = fx_exp2(u[j]);
#pragma unroll
                for (int ty = 0; ty < TX; ++ty)
#pragma unroll
                    for (int tx = 0; tx < TX; ++tx)
                        if (gy >= 32 * ty && gy <= 32 * ty + 33 && gx >= 32 * tx && gx <= 32 * tx + 33)
                            ex[ty * TX + tx] = max(ex[ty * TX + tx], e);
            }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const int m = __reduce_max_sync(0xffffffffu, ex[t]);
                if (lane == 0 && m > 0) atomicMax(&own_ex[t], m);
            }
            __syncthreads();
            if (tid < NT * CS) atomicMax(cl.map_shared_rank(&all_ex[par][tid % NT], tid / NT), own_ex[tid % NT]);
            auto bar = cl.barrier_arrive();
            // meanwhile f - k^2 u on the own nodes
            double2 gv[NPT];
#pragma unroll
            for (int j = 0; j < NPT; ++j) {
                const int wy = (tid + j * TNT) / S;
                if (wy < 1 || wy > RB) continue;
                gv[j] = make_double2(fma(u[j].x, mk2, fv[j].x), fma(u[j].y, mk2, fv[j].y));
            }
            cl.barrier_wait(std::move(bar));
            // r_{N+1} on the band's own nodes, into every CTA's right-hand side
#pragma unroll
            for (int j = 0; j < NPT; ++j) {
                const int q = tid + j * TNT, wy = q / S, gx = q - wy * S, gy = row0 - 1 + wy;
                if (q >= Y::WN || wy < 1 || wy > RB || gy > N0 || gx < 1 || gx > N0) continue;
                const int em = fx_scale(all_ex[par][((gy - 1) >> 5) * TX + ((gx - 1) >> 5)]);
                double2 r = make_double2(fx_nan(), fx_nan());
                if (em >= 0)
                    r = helm_resid2d_g<DAMP>(u[j], fx_fix2(u[j], em), fx_fix2(U[q - 1], em), fx_fix2(U[q + 1], em),
                                             fx_fix2(U[q - S], em), fx_fix2(U[q + S], em), gv[j], mih2, damp, em);
                const float2 ri = Inner<float>::from(r);
                float2* const o = Rr + gy * S + ix<N0>(gx);
#pragma unroll
                for (int c = 0; c < CS; ++c) *cl.map_shared_rank(o, c) = ri;
            }
            cl.sync();
            // norms in k_residual2d's order: warp w of a 32 x 32 tile sums its rows w, w + 8,
            // ..., the warps of a tile and then the tiles are summed in FP64
            if (warp < 8 * NT) {
                const int t = warp >> 3, w = warp & 7;
                const int gx = 32 * (t % TX) + lane + 1;
                float r2 = 0.f, em2 = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int gy = 32 * (t / TX) + w + 8 * k + 1;
                    if (gx > N0 || gy > N0) continue;
                    r2 += abs2(Rr[gy * S + ix<N0>(gx)]);
                    em2 = fmaxf(em2, abs2(E[gy * S + ix<N0>(gx)]));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    r2 += __shfl_xor_sync(0xffffffffu, r2, o);
                    em2 = fmaxf(em2, __shfl_xor_sync(0xffffffffu, em2, o));
                }
                if (lane == 0) {
                    sa[warp] = r2;
                    sm[warp] = em2;
                }
            }
            __syncthreads();
            if (warp == 0) {
                double a = 0.0;
                float mf = 0.f;
                if (lane < NT) {
                    a = sum_floats(sa + 8 * lane, 8);
                    for (int w = 0; w < 8; ++w) mf = fmaxf(mf, sm[8 * lane + w]);
                }
#pragma unroll
                for (int o = NT / 2; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
                }
                if (lane == 0) {
                    pend_n[npend] = a;
                    pend_m[npend] = widen_any(mf);
                }
                ++npend;
                const long long a2 = __shfl_sync(0xffffffffu, __double_as_longlong(a), 0);
                const int N = it0 + done + 1;
                // squared norms are non-negative, so their bits order as they do.  Below the
                // last one (by more than the roots' and quotients' rounding) and above the
                // target the step only goes on: relres fell, it is finite and under 1e4
                const bool on = a2 + 64 < prev2 && a2 > conv2 && N < I.max_outer && npend < 32;
                prev2 = a2;
                __syncwarp();
                if (!on || done + 1 >= budget) {
                    double rel = 0.0;
                    if (lane < npend) {
                        rel = sqrt(pend_n[lane]) / sst.norm0;
                        const int Ni = N - npend + 1 + lane;
                        if (rank == 0) {
                            I.hist[Ni] = rel;
                            I.einf[Ni - 1] = sqrt(pend_m[lane]);
                        }
                    }
                    // the steps that went on leave run = 0 and their smallest (last) relres
                    const double before = __shfl_sync(0xffffffffu, rel, max(npend - 2, 0));
                    const double last = __shfl_sync(0xffffffffu, rel, npend - 1);
                    if (lane == 0) {
                        InstState s = sst;
                        if (npend > 1) {
                            s.run = 0;
                            s.prev = before;
                            s.rmin = fmin(s.rmin, before);
                        }
                        s.it = N;
                        status_rule(I, s, last, N, false);
                        sst = s;
                    }
                    npend = 0;
                }
            }
            __syncthreads();
            ++done;
            par ^= 1;
            if (sst.status != HELM_ST_ACTIVE || done >= budget) break;
        }
        // the iterate (and, for a later call, the right-hand side) back to global memory
        double2* __restrict__ uout = I.u[sst.it & 1];
        float2* __restrict__ grw = (float2*)lev_rhs(L0, 0, sst.it);
#pragma unroll
        for (int j = 0; j < NPT; ++j) {
            const int q = tid + j * TNT, wy = q / S, gx = q - wy * S, gy = row0 - 1 + wy;
            if (q >= Y::WN || wy < 1 || wy > RB || gy > N0 || gx < 1 || gx > N0) continue;
            uout[gy * S + gx] = u[j];
            grw[(size_t)gy * L0.pitch + gx] = Rr[gy * S + ix<N0>(gx)];
        }
        cl.sync();                                        // the neighbours' last reads of this CTA
    }
    if (rank != 0) return;
    // step control: the steps made are the largest count of the launch's instances
    if (tid == 0) {
        if (done > 0) st[item.inst] = sst;
        atomicMax(&ctl.ctrl[4], done);
        __threadfence();
        s_last = (atomicAdd(&ctl.ctrl[3], 1) == ctl.ninst - 1);
        if (s_last) {
            __threadfence();
            ctl.ctrl[0] += atomicExch(&ctl.ctrl[4], 0);
            ctl.ctrl[2] = 0;                              // each instance has finished or used the budget
            ctl.ctrl[3] = 0;
        }
    }
}

// can a cluster of this form be resident? (its attributes set, and the driver's own answer)
template <int N0, int CS, bool DAMP>
bool small_resident()
{
    const int b = (int)SmallLay<N0, CS>::BYTES;
    if (cudaFuncSetAttribute(k_small2d<N0, CS, DAMP>, cudaFuncAttributeMaxDynamicSharedMemorySize, b) != cudaSuccess ||
        max_carveout(k_small2d<N0, CS, DAMP>) != cudaSuccess)
        return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS);
    cfg.blockDim = dim3(TNT);
    cfg.dynamicSmemBytes = b;
    int clusters = 0;
    return cudaOccupancyMaxActiveClusters(&clusters, k_small2d<N0, CS, DAMP>, &cfg) == cudaSuccess && clusters > 0;
}
template <int N0, int CS> bool small_ok() { return small_resident<N0, CS, false>() && small_resident<N0, CS, true>(); }

template <int N0, int CS>
cudaError_t small_launch(const InstDesc* insts, InstState* st, const MgItem* items, int nitems, int nu1, int nu2,
                         int cycles, int damp, const StepCtl& ctl, cudaStream_t s)
{
    const size_t b = SmallLay<N0, CS>::BYTES;
    if (damp)
        launch_k(k_small2d<N0, CS, true>, dim3(CS * nitems), dim3(TNT), b, s, insts, st, items, nu1, nu2, cycles,
                 tail_table_2d(), ctl);
    else
        launch_k(k_small2d<N0, CS, false>, dim3(CS * nitems), dim3(TNT), b, s, insts, st, items, nu1, nu2, cycles,
                 tail_table_2d(), ctl);
    return cudaGetLastError();
}

}  // namespace

namespace {
// per device: the forms that fit it (bits of small2d_pick) with SMALL_KNOWN; 0: not asked yet
constexpr int SMALL_KNOWN = 1 << 8;
std::atomic<int> g_small[64];
}  // namespace

void setup_small2d()
{
    // once per device (the attributes are the kernels', not a plan's)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64 || g_small[dev].load()) {
        cudaGetLastError();
        return;
    }
    const int fits = (small_ok<63, 8>() ? SMALL_63_8 : 0) | (small_ok<63, 4>() ? SMALL_63_4 : 0) |
                     (small_ok<63, 2>() ? SMALL_63_2 : 0) | (small_ok<31, 4>() ? SMALL_31_4 : 0) |
                     (small_ok<31, 2>() ? SMALL_31_2 : 0);
    cudaGetLastError();
    g_small[dev] = fits | SMALL_KNOWN;
}

int small2d_fits(int n, int ninst, bool mixed)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) {
        cudaGetLastError();
        return 0;
    }
    return small2d_pick(n, ninst, mixed, g_small[dev].load());
}

cudaError_t launch_small2d(const InstDesc* insts, InstState* st, const MgItem* items, int nitems, int n, int cs,
                           int nu1, int nu2, int cycles, int damp, int* ctrl, cudaStream_t s)
{
    const StepCtl c{ctrl, 0, nitems, 0, 0};
    if (n == 63 && cs == 8) return small_launch<63, 8>(insts, st, items, nitems, nu1, nu2, cycles, damp, c, s);
    if (n == 63 && cs == 4) return small_launch<63, 4>(insts, st, items, nitems, nu1, nu2, cycles, damp, c, s);
    if (n == 63 && cs == 2) return small_launch<63, 2>(insts, st, items, nitems, nu1, nu2, cycles, damp, c, s);
    if (n == 31 && cs == 4) return small_launch<31, 4>(insts, st, items, nitems, nu1, nu2, cycles, damp, c, s);
    if (n == 31 && cs == 2) return small_launch<31, 2>(insts, st, items, nitems, nu1, nu2, cycles, damp, c, s);
    return cudaErrorInvalidValue;
}

}  // namespace helm
