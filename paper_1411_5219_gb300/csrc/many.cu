// qcd_solve_cg_many: even-odd CG solves of several systems -- each with its
// own gauge field, lattice volume, hopping parameter, twisted mass and
// tolerance -- advanced together by ONE persistent kernel launch.
//
// The paper's finite-temperature studies are many independent runs over
// couplings and lattice sizes, a naturally parallel setup (Sec. 1), bounded
// by device memory (Sec. 2).  For small volumes one solve cannot fill the
// GPU: a launch's fixed cost and the latency of each thread's FP64 work set
// the time, not bandwidth.  Here a cooperative grid stays resident for the
// whole solve of every system: source preparation, the CG iterations on
// Mhat^dag Mhat x_e = Mhat^dag b'_e, the FP64 true-residual check, the odd-
// site reconstruction and the full-system residual, with barriers over a
// system's blocks between its phases instead of kernel launches.
//
// * Blocks are divided among the systems in proportion to their site
//   counts (at least one each).  Reductions are summed per fixed chunk of
//   work items and the chunks in a fixed order, so every sum -- and every
//   result -- is bitwise the same alone and in any batch.
// * Hopping phases use sixteen threads per site, one hop and one spin each,
//   in fixed point (fix_lanes.cuh); where the links do not fit that form,
//   eight threads per site in FP64 (hop_lanes.cuh).  Bound by latency: at
//   8^3 x 4 an iteration takes 38 us for six phases of one pass each (42 us
//   when each barrier read its generation, the error flag and the status from
//   memory).  Twelve systems of 432 to 5184 sites per parity: 17.4 ms with FP64
//   phases, one barrier over all blocks and its last block adding up every
//   system in turn; 10.8 ms with the fixed-point phases; 7.7 ms with a barrier
//   per system, whose last block sums that system alone.
// * Every barrier wait is bounded by a clock64 budget.  When it runs out the
//   kernel records QCD_ERR_TIMEOUT and every block returns; the call then
//   fails with that status and the context stays usable.
//
// Conventions as in the other kernels (chiral basis, D_hop with (1 - gamma)
// forward and (1 + gamma) backward, A = 1 + i a gamma_5, a = 2 kappa mu,
// antiperiodic t through t_bc).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "qcd_handles.h"
#include "fix_lanes.cuh"

namespace qcd {
namespace {

#define QCD_CHECK_CUDA(expr, what)                        \
    do {                                                  \
        cudaError_t e_ = (expr);                          \
        if (e_ != cudaSuccess) return check_cuda(e_, what); \
    } while (0)

constexpr int kManyThreads = 128;
constexpr int kManyMax = 32;

// A half field of FP64 spinors: 12 planes of double2, site-fastest.
struct HV {
    double2 *d;
    int stride;
};

// Coefficients of one hopping phase: out = cy[chi] y + cd[chi] (D in).
struct PhaseCoef {
    double cy[2][2], cd[2][2];
};

enum ManyPhaseCoef : int {
    MC_SRC_B = 0,   // b' = b_e + kappa D_eo t               (cy = 1, cd = kappa)
    MC_SRC_T,       // t = A^-dag D_oe^dag b'               (cy = 0, cd = A^-dag)
    MC_SRC_R,       // rhs = A^dag b' - kappa^2 D_eo^dag t  (cy = A^dag, cd = -kappa^2)
    MC_OP1,         // t = A^-1 D_oe p
    MC_OP2,         // s = A p - kappa^2 D_eo t
    MC_OP3,         // t = A^-dag D_oe^dag s
    MC_OP4,         // q = A^dag s - kappa^2 D_eo^dag t
    MC_RECON,       // x_o = A^-1 b_o + kappa A^-1 D_oe x_e
    MC_FULL,        // M x = A x - kappa D x
    MC_COUNT
};

struct ManySys {
    Geom g;
    const double2 *U;   // FP64 reconstruct-18 links: block (parity*4 + mu), 9 planes each
    int ustride;
    const int4 *fix;    // the links in fixed point (fixed.cuh), or nullptr
    HV be, bo, xe, xo;  // the caller's b and x
    HV bp, rhs, r, p, q, t, s;
    double tw_inv[2][2];    // A^-1 per chirality (source preparation)
    PhaseCoef pc[MC_COUNT];
    double tol2;
    int block0, nblocks;  // this system's blocks
    int chunk0;           // offset of its reduction chunks in each partial slot
};

enum ManyStatus : int { MS_RUNNING = 0, MS_CONVERGED = 1, MS_DONE = 2, MS_BREAKDOWN = 3, MS_MAXITER = 4 };

struct alignas(128) ManySysState {
    double b2, rr, pAp, alpha, beta, rr_stop, rr_true, full_r2, full_b2;
    int status;
    int iter;              // CG iterations
    int reliable;          // true-residual passes
    unsigned arrive;       // arrivals at this system's barrier (zero at launch)
    unsigned gen;          // barriers passed
};

struct ManyState {
    ManySysState s[kManyMax];
    int maxiter;
    int error;             // QCD_ERR_TIMEOUT when a barrier wait ran out
    int timeout_where;     // phase index of the first timeout
};

// ---- a system's barrier with a finaliser run by its last block to arrive
//
// Reductions are summed per chunk of kManyThreads consecutive work items of
// a system (whichever block processes the chunk writes its partial), and
// the finaliser adds the system's chunks with the whole block in a fixed
// order.  The result therefore depends neither on how many blocks a system
// gets nor on what else is in the batch.

struct Ctx {
    const ManySys *sys;
    ManyState *st;
    double *part;          // [slot][chunk] partials
    int nchunk;            // chunks per slot (all systems)
    long long budget;      // clock64 cycles a barrier wait may take
};

// Sum of this block's v (thread 0 gets it), fixed order.
__device__ __forceinline__ double block_total(double v)
{
    __shared__ double sm[32];
    double a[1] = {v};
    block_sum<1>(a, sm);
    return a[0];
}

// A system's total of the chunk partials in `slot` (items_per_site work
// items per site); every thread of the block calls it, thread 0 gets it.
__device__ __forceinline__ double chunk_sum(const Ctx &x, int slot, int k, int items_per_site)
{
    const ManySys &S = x.sys[k];
    const int nc = (S.g.h * items_per_site + kManyThreads - 1) / kManyThreads;
    const double *p = x.part + (size_t)slot * x.nchunk + S.chunk0;
    double a = 0.0;
    for (int c = threadIdx.x; c < nc; c += blockDim.x) a += __ldcg(p + c);
    return block_total(a);
}

// Barrier number `where` (0, 1, ...) over the blocks of system k; the systems
// do not wait for one another.  Before it, each block has written its chunk
// partials for this phase; the last block to arrive runs `fin` with all its
// threads (sums, CG decisions by thread 0), then releases the others.
// Returns false when the wait ran out, here or in another block (the kernel
// must return).  The generation is the barrier's number, known to every block,
// and the error flag is read while waiting only: each read of global memory
// that all blocks wait for costs a third of a microsecond.
template <typename Fin>
__device__ bool sys_barrier(const Ctx &x, int k, int where, Fin fin)
{
    __shared__ int ok, last;
    ManySysState &q = x.st->s[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        __threadfence();
        last = atomicAdd(&q.arrive, 1u) == (unsigned)x.sys[k].nblocks - 1;
    }
    __syncthreads();
    if (last) {
        __threadfence();
        fin();
        __syncthreads();
        if (threadIdx.x == 0) {
            q.arrive = 0;
            __threadfence();
            *(volatile unsigned *)&q.gen = (unsigned)where + 1u;
        }
    } else if (threadIdx.x == 0) {
        volatile unsigned *genp = &q.gen;
        const long long t0 = clock64();
        for (unsigned poll = 0; *genp != (unsigned)where + 1u; ++poll) {
            const bool out = clock64() - t0 > x.budget;
            if (out || ((poll & 15u) == 15u && *(volatile int *)&x.st->error != 0)) {
                if (atomicCAS(&x.st->error, 0, QCD_ERR_TIMEOUT) == 0) x.st->timeout_where = where;
                ok = 0;
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// ---- phases

// One complex component v of the output of a hopping phase: epilogue, store
// (or, without `out`, the difference from b), and what it adds to the sum.
__device__ __forceinline__ double hop_out(const ManySys &S, const PhaseCoef &pc, HV ManySys::*y, HV ManySys::*out, int p,
                                          int plane, int i, cx<double> v, bool norm)
{
    const int chi = plane / 6;
    v = cmul(mk(pc.cd[chi][0], pc.cd[chi][1]), v);
    if (y) {
        const double2 yy = __ldcg((S.*y).d + (size_t)plane * (S.*y).stride + i);
        v = cmac(v, mk(pc.cy[chi][0], pc.cy[chi][1]), mk(yy.x, yy.y));
    }
    if (!out) {
        // full residual: |b - M x|^2 (b of this parity)
        const HV &bh = p == 0 ? S.be : S.bo;
        const double2 bb = __ldg(bh.d + (size_t)plane * bh.stride + i);
        const double dr = bb.x - v.re, di = bb.y - v.im;
        return dr * dr + di * di;
    }
    const HV &o = S.*out;
    o.d[(size_t)plane * o.stride + i] = make_double2(v.re, v.im);
    return norm ? v.re * v.re + v.im * v.im : 0.0;
}

// Threads per site of a system's hopping phases.
__device__ __forceinline__ int hop_threads(const ManySys &S) { return S.fix ? 16 : 8; }

// A hopping phase: for every system, out (parity p) = cy y + cd D in on the
// system's blocks, sixteen threads per site in fixed point, eight in FP64;
// optionally |out|^2 -> slot.  Without `out`, |b - that|^2 is reduced and
// nothing is stored.
__device__ void hop_phase(const Ctx &x, int k, int lb, int coef, int p, bool dagger, HV ManySys::*in, HV ManySys::*y,
                          HV ManySys::*out, int red_slot)
{
    const ManySys &S = x.sys[k];
    const PhaseCoef &pc = S.pc[coef];
    // (copies: a store through a field would have the compiler load the
    // descriptor again in every pass of the loop)
    const Geom g = S.g;
    const int4 *const fix = S.fix;
    const int us = S.ustride, nblocks = S.nblocks, chunk0 = S.chunk0;
    const PlaneLoad<true> load{(S.*in).d, (S.*in).stride};
    const int items = g.h * (fix ? 16 : 8);
    for (int base = lb * kManyThreads; base < items; base += nblocks * kManyThreads) {
        const int w = base + threadIdx.x;
        const bool act = w < items;
        double red = 0.0;
        if (fix) {
            const int i = (act ? w : items - 1) >> 4, lane = w & 15;
            int E;
            i64 re, im;
            hop_fix16(g, fix, us, load, p, i, lane, dagger, E, re, im);
            if (act && (lane & 3) < 3) {
                const int plane = 6 * ((lane >> 2) & 1) + 3 * (lane >> 3) + (lane & 3);
                cx<double> v = mk(fix_value(re, E), fix_value(im, E));
                if (E == kFixRaw) {
                    double2 t[12];
                    hop_site_f64(g, fix, us, load, p, i, dagger, t);
                    v = mk(t[plane].x, t[plane].y);
                }
                red = hop_out(S, pc, y, out, p, plane, i, v, red_slot >= 0);
            }
        } else {
            const int i = w >> 3, lane = w & 7;
            cx<double> acc[12];
            if (act) {
                hop_lane8<true>(g, S.U, us, load.d, load.stride, p, i, lane, dagger, acc);
            } else {
#pragma unroll
                for (int a = 0; a < 12; ++a) acc[a] = mk(0.0, 0.0);
            }
            reduce_lanes8(acc, lane);
            if (act && !(lane & 1)) {
                const int spin = ((lane >> 2) << 1) | ((lane >> 1) & 1);
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    red += hop_out(S, pc, y, out, p, 3 * spin + a, i, acc[a], red_slot >= 0);
            }
        }
        if (red_slot >= 0) {
            const double t = block_total(red);
            if (threadIdx.x == 0) x.part[(size_t)red_slot * x.nchunk + chunk0 + base / kManyThreads] = t;
        }
    }
}

// |b|^2 of a full system (slot), for the full-residual statistics.
__device__ void bnorm_phase(const Ctx &x, int k, int lb, int slot)
{
    const ManySys &S = x.sys[k];
    const int items = S.g.h * 24;  // both parities, 12 complex each
    for (int base = lb * blockDim.x; base < items; base += S.nblocks * blockDim.x) {
        const int w = base + threadIdx.x;
        double red = 0.0;
        if (w < items) {
            const int par = w / (S.g.h * 12), r = w - par * S.g.h * 12, plane = r / S.g.h, i = r - plane * S.g.h;
            const HV &bh = par == 0 ? S.be : S.bo;
            const double2 v = __ldg(bh.d + (size_t)plane * bh.stride + i);
            red = v.x * v.x + v.y * v.y;
        }
        const double t = block_total(red);
        if (threadIdx.x == 0) x.part[(size_t)slot * x.nchunk + S.chunk0 + base / blockDim.x] = t;
    }
}

// Site-local vector phases, one thread per (site, complex component).
enum VecOp : int { V_TWIST_BO, V_SETUP, V_XR, V_P, V_TRUE, V_RESTART };

__device__ void vec_phase(const Ctx &x, int k, int lb, VecOp op, int red_slot)
{
    const ManySys &S = x.sys[k];
    const ManySysState &q = x.st->s[k];
    const int status = __ldcg(&q.status);
    const bool running = status == MS_RUNNING;
    const bool conv = status == MS_CONVERGED;
    bool go = true;
    if (op == V_XR || op == V_P) go = running;
    if (op == V_TRUE || op == V_RESTART) go = conv;
    if (go) {
        const int items = S.g.h * 12;
        for (int base = lb * blockDim.x; base < items; base += S.nblocks * blockDim.x) {
            const int w = base + threadIdx.x;
            double red = 0.0;
            const int plane = w / S.g.h, i = w - plane * S.g.h;
            auto at = [&](const HV &f) { return f.d + (size_t)plane * f.stride + i; };
            if (w < items) {
            // fields written earlier in this launch are read through L2 (__ldcg):
            // another SM's L1 may hold an older copy
            if (op == V_TWIST_BO) {  // t = A^-1 b_o (odd)
                const double2 b = __ldg(at(S.bo));
                const int chi = plane / 6;
                const cx<double> c = mk(S.tw_inv[chi][0], S.tw_inv[chi][1]), v = cmul(c, mk(b.x, b.y));
                *at(S.t) = make_double2(v.re, v.im);
            } else if (op == V_SETUP) {  // r = p = rhs, x_e = 0
                const double2 b = __ldcg(at(S.rhs));
                *at(S.r) = b;
                *at(S.p) = b;
                *at(S.xe) = make_double2(0.0, 0.0);
            } else if (op == V_XR) {  // x += alpha p, r -= alpha q, |r|^2
                const double a = __ldcg(&q.alpha);
                const double2 pp = __ldcg(at(S.p)), qq = __ldcg(at(S.q));
                double2 xx = __ldcg(at(S.xe)), rr = __ldcg(at(S.r));
                xx.x = fma(a, pp.x, xx.x);
                xx.y = fma(a, pp.y, xx.y);
                rr.x = fma(-a, qq.x, rr.x);
                rr.y = fma(-a, qq.y, rr.y);
                *at(S.xe) = xx;
                *at(S.r) = rr;
                red += rr.x * rr.x + rr.y * rr.y;
            } else if (op == V_P) {  // p = r + beta p
                const double bt = __ldcg(&q.beta);
                const double2 rr = __ldcg(at(S.r));
                double2 pp = __ldcg(at(S.p));
                pp.x = fma(bt, pp.x, rr.x);
                pp.y = fma(bt, pp.y, rr.y);
                *at(S.p) = pp;
            } else if (op == V_TRUE) {  // r = rhs - q (the FP64 true residual), |r|^2
                const double2 b = __ldcg(at(S.rhs)), qq = __ldcg(at(S.q));
                const double2 rr = make_double2(b.x - qq.x, b.y - qq.y);
                *at(S.r) = rr;
                red += rr.x * rr.x + rr.y * rr.y;
            } else {  // V_RESTART: p = r
                *at(S.p) = __ldcg(at(S.r));
            }
            }
            if (red_slot >= 0) {
                const double t = block_total(red);
                if (threadIdx.x == 0) x.part[(size_t)red_slot * x.nchunk + S.chunk0 + base / blockDim.x] = t;
            }
        }
    }
}

// ---- the persistent kernel

__global__ void __launch_bounds__(kManyThreads, 3) many_cg_kernel(const ManySys *sys, ManyState *st, double *part,
                                                                 const int *block_sys, int nchunk, long long budget)
{
    const Ctx x{sys, st, part, nchunk, budget};
    const int k = block_sys[blockIdx.x];
    const int lb = blockIdx.x - sys[k].block0;
    const int ht = hop_threads(sys[k]);
    ManySysState &q = st->s[k];
    int where = 0;
#define QCD_SYNC(FIN)                                        \
    if (!sys_barrier(x, k, where++, [&]() { FIN; })) return;
    // ---- source: t = A^-1 b_o ; b' = b_e + kappa D_eo t ; t = A^-dag D_oe^dag b' ;
    //      rhs = A^dag b' - kappa^2 D_eo^dag t (|rhs|^2) ; r = p = rhs, x_e = 0
    vec_phase(x, k, lb, V_TWIST_BO, -1);
    QCD_SYNC(;)
    hop_phase(x, k, lb, MC_SRC_B, 0, false, &ManySys::t, &ManySys::be, &ManySys::bp, -1);
    QCD_SYNC(;)
    hop_phase(x, k, lb, MC_SRC_T, 1, true, &ManySys::bp, nullptr, &ManySys::t, -1);
    QCD_SYNC(;)
    hop_phase(x, k, lb, MC_SRC_R, 0, true, &ManySys::t, &ManySys::bp, &ManySys::rhs, 0);
    QCD_SYNC({
        const double b2 = chunk_sum(x, 0, k, ht);
        if (threadIdx.x == 0) {
            q.b2 = q.rr = q.rr_true = b2;
            q.rr_stop = x.sys[k].tol2 * b2;
            q.alpha = q.beta = q.pAp = 0.0;
            q.status = b2 == 0.0 ? MS_DONE : (isfinite(b2) ? MS_RUNNING : MS_BREAKDOWN);
            q.iter = 0;
            q.reliable = 0;
        }
    })
    vec_phase(x, k, lb, V_SETUP, -1);
    QCD_SYNC(;)
    for (;;) {
        // the loop decision is read by every block after the same barrier
        const int status = __ldcg(&q.status);
        if (status == MS_RUNNING && __ldcg(&q.iter) < st->maxiter) {
            // ---- one CG iteration
            hop_phase(x, k, lb, MC_OP1, 1, false, &ManySys::p, nullptr, &ManySys::t, -1);
            QCD_SYNC(;)
            hop_phase(x, k, lb, MC_OP2, 0, false, &ManySys::t, &ManySys::p, &ManySys::s, 0);
            QCD_SYNC({
                const double pAp = chunk_sum(x, 0, k, ht);
                if (threadIdx.x == 0) {
                    q.pAp = pAp;
                    if (!(pAp > 0.0) || !isfinite(pAp)) {
                        q.status = MS_BREAKDOWN;
                        q.alpha = 0.0;
                    } else {
                        q.alpha = q.rr / pAp;
                    }
                }
            })
            hop_phase(x, k, lb, MC_OP3, 1, true, &ManySys::s, nullptr, &ManySys::t, -1);
            QCD_SYNC(;)
            hop_phase(x, k, lb, MC_OP4, 0, true, &ManySys::t, &ManySys::s, &ManySys::q, -1);
            QCD_SYNC(;)
            vec_phase(x, k, lb, V_XR, 0);
            QCD_SYNC({
                const double rn = chunk_sum(x, 0, k, 12);
                if (threadIdx.x == 0) {
                    q.iter += 1;
                    // another system's wait ran out and the call fails: a block that
                    // waits sees it there, the only block of a system has no waits
                    if (x.sys[k].nblocks == 1 && *(volatile int *)&x.st->error != 0) q.status = MS_BREAKDOWN;
                    if (q.status == MS_RUNNING) {
                        if (!isfinite(rn)) {
                            q.status = MS_BREAKDOWN;
                        } else {
                            q.beta = rn / q.rr;
                            q.rr = rn;
                            if (rn <= q.rr_stop) q.status = MS_CONVERGED;
                        }
                    }
                }
            })
            vec_phase(x, k, lb, V_P, -1);
            QCD_SYNC(;)
        } else if (status == MS_CONVERGED) {
            // ---- FP64 true residual: q = Mhat^dag Mhat x_e (via s, t), r = rhs - q;
            //      DONE if it meets the target, else CG restarts from it
            hop_phase(x, k, lb, MC_OP1, 1, false, &ManySys::xe, nullptr, &ManySys::t, -1);
            QCD_SYNC(;)
            hop_phase(x, k, lb, MC_OP2, 0, false, &ManySys::t, &ManySys::xe, &ManySys::s, -1);
            QCD_SYNC(;)
            hop_phase(x, k, lb, MC_OP3, 1, true, &ManySys::s, nullptr, &ManySys::t, -1);
            QCD_SYNC(;)
            hop_phase(x, k, lb, MC_OP4, 0, true, &ManySys::t, &ManySys::s, &ManySys::q, -1);
            QCD_SYNC(;)
            vec_phase(x, k, lb, V_TRUE, 0);
            QCD_SYNC({
                const double rt = chunk_sum(x, 0, k, 12);
                if (threadIdx.x == 0) {
                    q.reliable += 1;
                    q.rr_true = rt;
                    if (!isfinite(rt)) {
                        q.status = MS_BREAKDOWN;
                    } else if (rt <= q.rr_stop) {
                        q.status = MS_DONE;
                    } else {
                        // restart from the true residual (still CONVERGED for the next phase)
                        q.rr = rt;
                        q.beta = 0.0;
                    }
                }
            })
            vec_phase(x, k, lb, V_RESTART, -1);
            QCD_SYNC({
                if (threadIdx.x == 0 && q.status == MS_CONVERGED) q.status = MS_RUNNING;
            })
        } else {
            break;
        }
    }
    // ---- odd sites x_o = A^-1 b_o + kappa A^-1 D_oe x_e, then |b - M x|^2, |b|^2
    hop_phase(x, k, lb, MC_RECON, 1, false, &ManySys::xe, &ManySys::bo, &ManySys::xo, -1);
    QCD_SYNC(;)
    // M x per parity: out = A x - kappa D x (even from x_o, odd from x_e)
    hop_phase(x, k, lb, MC_FULL, 0, false, &ManySys::xo, &ManySys::xe, nullptr, 0);
    hop_phase(x, k, lb, MC_FULL, 1, false, &ManySys::xe, &ManySys::xo, nullptr, 1);
    bnorm_phase(x, k, lb, 2);
    QCD_SYNC({
        const double r0 = chunk_sum(x, 0, k, ht);
        const double r1 = chunk_sum(x, 1, k, ht);
        const double b2 = chunk_sum(x, 2, k, 24);
        if (threadIdx.x == 0) {
            q.full_r2 = r0 + r1;
            q.full_b2 = b2;
            if (q.status == MS_RUNNING || q.status == MS_CONVERGED) q.status = MS_MAXITER;
        }
    })
#undef QCD_SYNC
}

void put(PhaseCoef &pc, const Coef &cy, const Coef &cd)
{
    memcpy(pc.cy, cy.c, sizeof(pc.cy));
    memcpy(pc.cd, cd.c, sizeof(pc.cd));
}

}  // namespace
}  // namespace qcd

using namespace qcd;

static qcd_status solve_many(LinkWait wait, int n, const qcd_gauge *const *gauges, qcd_spinor *const *x,
                             const qcd_spinor *const *b, const qcd_solver_params *prm, qcd_solver_stats *stats,
                             long long wait_cycles, int max_blocks, void *stream)
{
    const auto t0 = std::chrono::steady_clock::now();
    if (n < 1 || n > kManyMax) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: n = %d not in 1..%d", n, kManyMax);
    if (!gauges || !x || !b || !prm) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: NULL argument");
    for (int k = 0; k < n; ++k) {
        const qcd_gauge *g = gauges[k];
        if (!g || !x[k] || !b[k]) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: NULL handle (system %d)", k);
        if (g->prec != QCD_PREC_F64) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: gauge field %d must be F64", k);
        // x and b live on the gauge field's lattice or on a context lattice of
        // the same extents (whose handle then holds this system's scratch)
        const qcd_lattice *xl = x[k]->lat;
        if (b[k]->lat != xl || memcmp(xl->dims, g->lat->dims, sizeof(xl->dims)) != 0 || xl->t_bc != g->lat->t_bc)
            return fail(QCD_ERR_INVALID_ARG,
                        "solve_cg_many: x and b of system %d must share a lattice with the gauge field's extents", k);
        if (x[k]->parity != QCD_PARITY_FULL || b[k]->parity != QCD_PARITY_FULL || x[k]->prec != QCD_PREC_F64 ||
            b[k]->prec != QCD_PREC_F64 || x[k]->ks || b[k]->ks)
            return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: x and b must be FULL F64 Wilson fields (system %d)", k);
        if (x[k]->data == b[k]->data) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: x aliases b (system %d)", k);
        for (int j = 0; j < k; ++j)
            if (x[j]->data == x[k]->data) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: systems %d and %d share x", j, k);
        const qcd_solver_params &q = prm[k];
        if (!q.eo || q.normal || q.inner_prec != QCD_PREC_F64)
            return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: even-odd FP64 CG only (eo = 1, normal = 0, inner F64; system %d)", k);
        if (!(q.tol > 0.0) || q.maxiter < 1 || q.maxiter > (1 << 30) || !std::isfinite(q.kappa) || !std::isfinite(q.mu))
            return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: bad tol/maxiter/kappa/mu (system %d)", k);
        if (q.maxiter != prm[0].maxiter)
            return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: the systems share one maxiter (system %d)", k);
    }
    if (wait_cycles < 0) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: wait_cycles must be >= 0");
    if (max_blocks < 0 || (max_blocks > 0 && max_blocks < n))
        return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: max_blocks = %d must be 0 or at least n = %d", max_blocks, n);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, nsm = 0, per_sm = 0, coop = 0;
    QCD_CHECK_CUDA(cudaGetDevice(&dev), "solve_cg_many");
    QCD_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev), "solve_cg_many");
    QCD_CHECK_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev), "solve_cg_many");
    if (!coop) return fail(QCD_ERR_CUDA, "solve_cg_many: the device has no cooperative launch");
    QCD_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, many_cg_kernel, kManyThreads, 0),
                   "solve_cg_many: occupancy");
    if (per_sm < 1) return fail(QCD_ERR_CUDA, "solve_cg_many: the kernel does not fit an SM");
    // blocks: every block resident (cooperative launch), divided among the
    // systems in proportion to their sites, at least one each, and no more
    // than a system can use (16 threads per site)
    long long total_h = 0;
    for (int k = 0; k < n; ++k) total_h += x[k]->lat->h;
    // every block resident at once; a caller sharing the GPU with other work
    // may ask for fewer (max_blocks), so the launch need not wait for the
    // whole GPU to drain
    const int grid_cap = max_blocks > 0 ? std::min(max_blocks, nsm * per_sm) : nsm * per_sm;
    std::vector<int> nb(n);
    int used = 0;
    for (int k = 0; k < n; ++k) {
        const int h = x[k]->lat->h;
        const int useful = std::max(1, (16 * h + kManyThreads - 1) / kManyThreads);
        nb[k] = std::max(1, std::min(useful, (int)((long long)(grid_cap - n) * h / total_h)));
        used += nb[k];
    }
    if (used > grid_cap) return fail(QCD_ERR_INVALID_ARG, "solve_cg_many: too many systems for one resident grid");
    std::vector<ManySys> hs(n);
    std::vector<int> block_sys;
    int nchunk = 0;  // reduction chunks per partial slot, all systems
    const qcd_lattice *lat0 = x[0]->lat;
    std::vector<HopLinks> links(n);  // (held until the solve is done)
    for (int k = 0; k < n; ++k) {
        const qcd_gauge *g = gauges[k];
        const qcd_lattice *lat = x[k]->lat;
        qcd_status st = QCD_OK;
        links[k] = hop_links(g, QCD_PREC_F64, g->recon, s, wait, &st);
        GaugeView U = links[k].form[0];
        if (st != QCD_OK) return st;
        if (!U.fix && g->recon != 18) U = gauge_view(g, QCD_PREC_F64, 18, s, &st);  // (the FP64 phases read all nine entries)
        if (st != QCD_OK) return st;
        ManySys &S = hs[k];
        memset(&S, 0, sizeof(S));
        S.g = lat->geom;
        S.U = static_cast<const double2 *>(U.data);
        S.ustride = U.stride;
        S.fix = U.fix;
        auto half = [&](const qcd_spinor *f, int h) {
            return HV{reinterpret_cast<double2 *>(static_cast<char *>(f->data) + h * f->half_data_bytes), lat->stride};
        };
        S.be = half(b[k], 0);
        S.bo = half(b[k], 1);
        S.xe = half(x[k], 0);
        S.xo = half(x[k], 1);
        const char *names[7] = {"bp", "rhs", "r", "p", "q", "t", "s"};
        HV *dst[7] = {&S.bp, &S.rhs, &S.r, &S.p, &S.q, &S.t, &S.s};
        for (int f = 0; f < 7; ++f) {
            const FieldView v = ws_field(lat, std::string("many") + std::to_string(k) + "_" + names[f], 1, QCD_PREC_F64);
            if (!v.hv[0].data) return fail(QCD_ERR_OOM, "solve_cg_many: workspace");
            *dst[f] = HV{static_cast<double2 *>(v.hv[0].data), v.hv[0].stride};
        }
        const double kappa = prm[k].kappa, a = 2.0 * kappa * prm[k].mu;
        const Coef zero = coef_real(0.0);
        memcpy(S.tw_inv, coef_twist_inv(a).c, sizeof(S.tw_inv));
        put(S.pc[MC_SRC_B], coef_real(1.0), coef_real(kappa));
        put(S.pc[MC_SRC_T], zero, coef_twist_inv(-a));
        put(S.pc[MC_SRC_R], coef_twist(-a), coef_real(-kappa * kappa));
        put(S.pc[MC_OP1], zero, coef_twist_inv(a));
        put(S.pc[MC_OP2], coef_twist(a), coef_real(-kappa * kappa));
        put(S.pc[MC_OP3], zero, coef_twist_inv(-a));
        put(S.pc[MC_OP4], coef_twist(-a), coef_real(-kappa * kappa));
        put(S.pc[MC_RECON], coef_twist_inv(a), coef_scale(coef_twist_inv(a), kappa));
        put(S.pc[MC_FULL], coef_twist(a), coef_real(-kappa));
        S.tol2 = prm[k].tol * prm[k].tol;
        S.block0 = (int)block_sys.size();
        S.chunk0 = nchunk;
        nchunk += (24 * lat->h + kManyThreads - 1) / kManyThreads;
        S.nblocks = nb[k];
        for (int j = 0; j < nb[k]; ++j) block_sys.push_back(k);
    }
    const int grid = (int)block_sys.size();
    // device-side descriptors, state and partials (workspace of the first
    // system's lattice; the host copies are staged in pageable memory and
    // the stream is synchronised before this call returns)
    const size_t desc_bytes = sizeof(ManySys) * n, bs_bytes = sizeof(int) * grid, st_bytes = sizeof(ManyState),
                 part_bytes = sizeof(double) * 3 * (size_t)nchunk;
    char *ws = static_cast<char *>(workspace(lat0, "many_ctl", desc_bytes + bs_bytes + st_bytes + part_bytes + 1024));
    if (!ws) return fail(QCD_ERR_OOM, "solve_cg_many: workspace");
    auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
    ManySys *d_sys = reinterpret_cast<ManySys *>(ws);
    int *d_bs = reinterpret_cast<int *>(ws + align(desc_bytes));
    ManyState *d_st = reinterpret_cast<ManyState *>(ws + align(desc_bytes) + align(bs_bytes));
    double *d_part = reinterpret_cast<double *>(ws + align(desc_bytes) + align(bs_bytes) + align(st_bytes));
    ManyState h_st;
    memset(&h_st, 0, sizeof(h_st));
    h_st.maxiter = prm[0].maxiter;
    QCD_CHECK_CUDA(cudaMemcpyAsync(d_sys, hs.data(), desc_bytes, cudaMemcpyHostToDevice, s), "solve_cg_many");
    QCD_CHECK_CUDA(cudaMemcpyAsync(d_bs, block_sys.data(), bs_bytes, cudaMemcpyHostToDevice, s), "solve_cg_many");
    QCD_CHECK_CUDA(cudaMemcpyAsync(d_st, &h_st, sizeof(h_st), cudaMemcpyHostToDevice, s), "solve_cg_many");
    long long budget = wait_cycles > 0 ? wait_cycles : 4000000000LL;  // ~2 s at 2 GHz
    int nc = nchunk;
    void *args[] = {&d_sys, &d_st, &d_part, &d_bs, &nc, &budget};
    QCD_CHECK_CUDA(cudaLaunchCooperativeKernel((const void *)many_cg_kernel, dim3(grid), dim3(kManyThreads), args, 0, s),
                   "solve_cg_many: launch");
    note_launches();
    QCD_CHECK_CUDA(cudaMemcpyAsync(&h_st, d_st, sizeof(h_st), cudaMemcpyDeviceToHost, s), "solve_cg_many");
    QCD_CHECK_CUDA(cudaStreamSynchronize(s), "solve_cg_many");
    if (h_st.error == QCD_ERR_TIMEOUT)
        return fail(QCD_ERR_TIMEOUT, "solve_cg_many: a grid barrier wait ran out of its %lld-cycle budget (phase %d)",
                    budget, h_st.timeout_where);
    qcd_status result = QCD_OK;
    const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    for (int k = 0; k < n; ++k) {
        const ManySysState &q = h_st.s[k];
        if (q.status == MS_BREAKDOWN)
            result = fail(QCD_ERR_BREAKDOWN, "solve_cg_many: breakdown in system %d", k);
        else if (q.status != MS_DONE && result == QCD_OK)
            result = fail(QCD_ERR_NOT_CONVERGED, "solve_cg_many: maxiter reached (system %d)", k);
        if (stats) {
            stats[k].iterations = q.iter;
            stats[k].reliable_updates = q.reliable;
            stats[k].true_rel_residual = q.b2 > 0.0 ? std::sqrt(q.rr_true / q.b2) : 0.0;
            stats[k].full_rel_residual = q.full_b2 > 0.0 ? std::sqrt(q.full_r2 / q.full_b2) : 0.0;
            stats[k].seconds = secs;
        }
    }
    return result;
}

extern "C" qcd_status qcd_solve_cg_many(int n, const qcd_gauge *const *gauges, qcd_spinor *const *x,
                                        const qcd_spinor *const *b, const qcd_solver_params *prm,
                                        qcd_solver_stats *stats, long long wait_cycles, int max_blocks,
                                        void *stream)
{
    const qcd_status st = solve_many(LINKS_SETTLE, n, gauges, x, b, prm, stats, wait_cycles, max_blocks, stream);
    if (st != QCD_ERR_OOM) return st;
    bool any = false;  // (as with_memory, for every system's field)
    for (int k = 0; k < n; ++k) any = give_back_fixed(gauges[k], x[k]->lat, static_cast<cudaStream_t>(stream)) || any;
    return any ? solve_many(LINKS_FP64, n, gauges, x, b, prm, stats, wait_cycles, max_blocks, stream) : st;
}
