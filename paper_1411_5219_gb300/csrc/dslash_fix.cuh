// The FP64 hopping kernel in fixed point (fixed.cuh): the
// launches, epilogues and fused reduction of dslash_kernel, with the input in
// fixed point and y and the output in either form.
#pragma once

#include "fix_lanes.cuh"

namespace qcd {

constexpr int kFixThreads = 128;  // two threads per element
constexpr int kFixElems = kFixThreads / 2;
constexpr int kFixStages = 2;     // hops staged in shared memory
constexpr int kFixSlot = (12 + 9) * 16;  // int4 of one hop of a warp's 16 elements: spinor components, link entries

__device__ __forceinline__ void copy16(int4 *dst, const int4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// Lanes 0-15 of a warp take spin 0 of the half spinors of 16 consecutive
// elements, lanes 16-31 spin 1: one thread per element needs 168 registers
// and more (400 us at 48^3 x 12), a thread pair shares the link loads of its
// warp and holds 36 registers of sums instead of 48.  Bound by memory latency
// next to HBM: with direct loads the compiler keeps no hop ahead in registers
// (250 us), so each warp copies the next hop's components and links to a
// two-slot ring in shared memory with cp.async while it multiplies this one
// (205 us for 1.05 GB, 76 % of HBM; the FP64 kernel took 938 us; a call with the
// conversion of an FP64 input takes 247 us).  Three slots
// at 12 warps per SM or two at 20 (96 registers, spills) measured slower than
// two at 16.
template <int kDagger, int kEpi, bool kReduce, typename Launch = DslashLaunch>
__global__ void __launch_bounds__(kFixThreads, 4) dslash_fix_kernel(const __grid_constant__ Launch a)
{
    constexpr bool kMulti = std::is_same<Launch, DslashMulti>::value;  // separate fields, consecutive blocks one each
    if (a.check_status && a.state->status != a.run_status) return;
    if (a.U.unfit && *a.U.unfit) return;
    constexpr int SF_ = kDagger ? -1 : +1, SB_ = -SF_;  // projector signs of forward and backward hops
    const int ne = a.g.h << a.rhs_log2;
    int nbp = (ne + kFixElems - 1) / kFixElems, field = 0;
    if constexpr (kMulti) nbp *= a.n;
    const int p = a.both ? (int)(blockIdx.x >= (unsigned)nbp) : a.out_parity;
    int bl = blockIdx.x - (a.both ? p * nbp : 0);
    if constexpr (kMulti) {
        field = bl % a.n;
        bl /= a.n;
    }
    if (a.tmap) bl = (bl % a.g.L[3]) * a.tmap + bl / a.g.L[3];
    const int spin = (threadIdx.x >> 4) & 1;
    const int e = bl * kFixElems + (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
    const int L = a.rhs_log2, rhs = e & ((1 << L) - 1);
    const bool act = e < ne;
    const int i = (act ? e : ne - 1) >> L;  // (the tail works on the last element and stores nothing)
    double red[1] = {0.0};
    const Geom &g = a.g;
    SpinorView inv = a.in[p], outv = a.out[p];
    if constexpr (kMulti) {
        inv = a.input(p, field);
        outv = a.output(p, field);
    }
    const size_t is = inv.stride, us = a.U.stride;
    const int4 *in = static_cast<const int4 *>(inv.data);
    const SiteCoords c = site_coords(g, i, p);
    const int base = i - c.xh;
    const bool wf = c.t == g.L[3] - 1, wb = c.t == 0, anti = antiperiodic(g);
    // neighbours in the order y+, y-, x+, x-, z+, z-, t+, t-
    const int nb[8] = {c.y == g.L[1] - 1 ? i - (g.L[1] - 1) * g.sy : i + g.sy,
                       c.y == 0 ? i + (g.L[1] - 1) * g.sy : i - g.sy,
                       base + ((c.x + 1 == g.L[0] ? 0 : c.x + 1) >> 1),
                       base + ((c.x == 0 ? g.L[0] - 1 : c.x - 1) >> 1),
                       c.z == g.L[2] - 1 ? i - (g.L[2] - 1) * g.sz : i + g.sz,
                       c.z == 0 ? i + (g.L[2] - 1) * g.sz : i - g.sz,
                       wf ? i - (g.L[3] - 1) * g.st : i + g.st,
                       wb ? i + (g.L[3] - 1) * g.st : i - g.st};
    int E[8], Em = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        E[k] = SpFix::exponent(inv, (nb[k] << L) | rhs);
        Em = max(Em, E[k]);
    }
    const int sg = spin ? -1 : 1;
    // Each warp stages its hops in a ring of its own: a lane copies the six
    // spinor components of its half of the planes and every other link
    // entry of its element.
    __shared__ int4 ring[kFixThreads / 32][kFixStages][kFixSlot];
    int4(&slots)[kFixStages][kFixSlot] = ring[threadIdx.x >> 5];
    const int el = threadIdx.x & 15;
    auto stage = [&](int k) {
        int4 *dst = slots[k % kFixStages] + el;
        const int4 *src = in + ((nb[k] << L) | rhs) + (size_t)(6 * spin) * is;
#pragma unroll
        for (int c = 0; c < 6; ++c) copy16(dst + (6 * spin + c) * 16, src + c * is);
        // mu of the hops in this order: y y x x z z t t
        const int mu = k < 2 ? 1 : k < 4 ? 0 : k / 2;
        const int4 *u = a.U.fix + (size_t)(((k & 1 ? 1 - p : p) * 4 + mu) * 9 + spin) * us + (k & 1 ? nb[k] : i);
#pragma unroll
        for (int c = 0; c < 4; ++c) copy16(dst + (12 + 2 * c + spin) * 16, u + 2 * c * us);
        if (spin == 0) copy16(dst + 20 * 16, u + 8 * us);
        asm volatile("cp.async.commit_group;");
    };
#pragma unroll
    for (int k = 0; k < kFixStages - 1; ++k) stage(k);
    FixAcc acc;
#define QCD_FIX(K, MU, S, ADJ, STAGE, FLIP)                                                              \
    {                                                                                                    \
        if ((K) + kFixStages - 1 < 8) stage(((K) + kFixStages - 1) & 7);                                 \
        asm volatile("cp.async.wait_group %0;" ::"n"((K) + kFixStages - 1 < 8 ? kFixStages - 1 : 7 - (K))); \
        __syncwarp();                                                                                    \
        const int4 *q = slots[(K) % kFixStages] + el;                                                    \
        hop_fix<MU, S, ADJ, STAGE, 16>(acc, q + 3 * spin * 16, q + ((MU) <= 1 ? 9 - 3 * spin : 6 + 3 * spin) * 16, \
                                       q + 12 * 16, sg, min(Em - E[K], 63), FLIP);                       \
        __syncwarp();                                                                                    \
    }
    QCD_FIX(0, 1, SF_, false, 0, false)
    QCD_FIX(1, 1, SB_, true, 1, false)
    negate_all(acc.lb, spin);
    QCD_FIX(2, 0, SF_, false, 1, false)
    QCD_FIX(3, 0, SB_, true, 1, false)
    QCD_FIX(4, 2, SF_, false, 1, false)
    QCD_FIX(5, 2, SB_, true, 2, false)
    negate_all(acc.la, spin);
    QCD_FIX(6, 3, SF_, false, 2, anti && wf)
    QCD_FIX(7, 3, SB_, true, 2, anti && wb)
#undef QCD_FIX
    // the other thread's x and y hops belong to this thread's lower spin
#pragma unroll
    for (int k = 0; k < 6; ++k) acc.la[k] += __shfl_xor_sync(0xffffffffu, acc.lb[k], 16);
    const bool raw = Em == kFixRaw, out_fix = a.out_fix;
    if (kEpi == EPI_PLAIN && out_fix && !__any_sync(0xffffffffu, raw)) {
        // D psi itself, in fixed point: the site's sums shifted to 56 bits
        unsigned long long top = 0ull;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            top |= (unsigned long long)(acc.up[k] ^ (acc.up[k] >> 63));
            top |= (unsigned long long)(acc.la[k] ^ (acc.la[k] >> 63));
        }
        top |= __shfl_xor_sync(0xffffffffu, top, 16);
        const int sh = max(64 - __clzll((long long)top) - kFixBits, 0);
        if (act) {
            int4 *o = static_cast<int4 *>(outv.data) + e;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const i64 *v = (k < 3 ? acc.up : acc.la) + 2 * (k % 3);
                int4 q;
                to_limbs(v[0] >> sh, q.x, q.y);
                to_limbs(v[1] >> sh, q.z, q.w);
                o[(size_t)((k < 3 ? 0 : 3) + 3 * spin + k) * outv.stride] = q;
            }
            if (spin == 0) reinterpret_cast<int *>(outv.norm)[e] = top == 0ull ? 0 : Em + sh;
        }
        return;
    }
    double d[12];  // D psi: re, im of three colours of spin s, then of spin 2 + s
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        d[k] = fix_value(acc.up[k], Em);
        d[6 + k] = fix_value(acc.la[k], Em);
    }
    if (raw) {
        double2 t[12];
        hop_site_f64(g, a.U.fix, a.U.stride, FixLoad{inv, L, rhs}, p, i, kDagger != 0, t);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 v = t[(k < 3 ? 0 : 3) + 3 * spin + k];
            d[2 * k] = v.x;
            d[2 * k + 1] = v.y;
        }
    }
    // epilogue, with coefficients from the kernel parameters or the device table of a CG
    const double *cf = a.coef ? a.coef + (size_t)rhs * a.coef_stride : nullptr;
    if (kEpi != EPI_PLAIN && act) {
        const int yE = (kEpi == EPI_REAL_YD || kEpi == EPI_CPLX_YD) && a.y_fix ? SpFix::exponent(a.y[p], e) : 0;
#pragma unroll
        for (int chi = 0; chi < 2; ++chi) {
            const cx<double> cd = mk(cf ? __ldg(cf + 4 + 2 * chi) : a.cd[chi][0], cf ? __ldg(cf + 5 + 2 * chi) : a.cd[chi][1]);
            const cx<double> cy = mk(cf ? __ldg(cf + 2 * chi) : a.cy[chi][0], cf ? __ldg(cf + 1 + 2 * chi) : a.cy[chi][1]);
            const size_t at = (size_t)(6 * chi + 3 * spin) * a.y[p].stride + e;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                cx<double> v = mk(d[6 * chi + 2 * k], d[6 * chi + 2 * k + 1]);
                if (kEpi == EPI_CPLX_D) {
                    v = cmul(cd, v);
                } else {
                    const int4 q = __ldg(static_cast<const int4 *>(a.y[p].data) + at + (size_t)k * a.y[p].stride);
                    const double2 y = fix_load(q, a.y_fix ? yE : kFixRaw);
                    v = fix_epilogue<kEpi == EPI_REAL_YD>(v, y, cy, cd);
                }
                d[6 * chi + 2 * k] = v.re;
                d[6 * chi + 2 * k + 1] = v.im;
            }
        }
    }
    int Eo = kFixRaw;
    if (out_fix) {
        unsigned top = 0u, low = 0u;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            top = max(top, twice_hi(d[k]));
            low |= (unsigned)__double2loint(d[k]);
        }
        top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
        low |= __shfl_xor_sync(0xffffffffu, low, 16);
        Eo = fix_exponent(top, low);
        if (act && spin == 0) reinterpret_cast<int *>(outv.norm)[e] = Eo;
    }
    if (act) {
        int4 *o = static_cast<int4 *>(outv.data) + e;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            // (kFixRaw: the FP64 form)
            o[(size_t)((k < 3 ? 0 : 3) + 3 * spin + k) * outv.stride] = fix_store(d[2 * k], d[2 * k + 1], Eo);
            if (kReduce) red[0] = fma(d[2 * k], d[2 * k], fma(d[2 * k + 1], d[2 * k + 1], red[0]));
        }
    }
    if (kReduce) {
        if (L == 5) {
            // 32 right-hand sides: a warp holds 16 of them, twice
            red[0] += __shfl_xor_sync(0xffffffffu, red[0], 16);
            if (spin != ((int)(threadIdx.x >> 5) & 1)) red[0] = 0.0;
        }
        grid_reduce_rhs<1>(red, a.rhs_log2, a.red, a.fin, a.state, a.red_out);
    }
}

// The hop of small lattices, sixteen threads per site (fix_lanes.cuh), FP64
// fields in and out.
template <int kEpi, bool kReduce>
__global__ void __launch_bounds__(128) dslash_fix16_kernel(const DslashLaunch a)
{
    if (a.check_status && a.state->status != a.run_status) return;
    if (a.U.unfit && *a.U.unfit) return;
    const int items = a.g.h * 16;
    const int nbp = (items + 127) / 128;
    const int p = a.both ? (int)(blockIdx.x >= (unsigned)nbp) : a.out_parity;
    const int w = (blockIdx.x - (a.both ? p * nbp : 0)) * 128 + threadIdx.x;
    const bool act = w < items;
    const int i = (act ? w : items - 1) >> 4, lane = w & 15;
    const PlaneLoad<false> load{static_cast<const double2 *>(a.in[p].data), a.in[p].stride};
    int E;
    i64 re, im;
    hop_fix16(a.g, a.U.fix, a.U.stride, load, p, i, lane, a.dagger != 0, E, re, im);
    double red[1] = {0.0};
    if (act && (lane & 3) < 3) {
        const int chi = (lane >> 2) & 1, plane = 6 * chi + 3 * (lane >> 3) + (lane & 3);
        cx<double> v = mk(fix_value(re, E), fix_value(im, E));
        if (E == kFixRaw) {
            double2 t[12];
            hop_site_f64(a.g, a.U.fix, a.U.stride, load, p, i, a.dagger != 0, t);
            v = mk(t[plane].x, t[plane].y);
        }
        const double *cf = a.coef;
        const cx<double> d = mk(cf ? __ldg(cf + 4 + 2 * chi) : a.cd[chi][0], cf ? __ldg(cf + 5 + 2 * chi) : a.cd[chi][1]);
        const cx<double> cy = mk(cf ? __ldg(cf + 2 * chi) : a.cy[chi][0], cf ? __ldg(cf + 1 + 2 * chi) : a.cy[chi][1]);
        if (kEpi == EPI_CPLX_D) {
            v = cmul(d, v);
        } else if (kEpi == EPI_REAL_YD || kEpi == EPI_CPLX_YD) {
            const double2 y = __ldg(static_cast<const double2 *>(a.y[p].data) + (size_t)plane * a.y[p].stride + i);
            v = fix_epilogue<kEpi == EPI_REAL_YD>(v, y, cy, d);
        }
        static_cast<double2 *>(a.out[p].data)[(size_t)plane * a.out[p].stride + i] = make_double2(v.re, v.im);
        red[0] = fma(v.re, v.re, v.im * v.im);
    }
    if (kReduce) grid_reduce_rhs<1>(red, 0, a.red, a.fin, a.state, a.red_out);
}

inline cudaError_t launch_dslash_fix16(const DslashLaunch &a, cudaStream_t s)
{
    if (a.rhs_log2 != 0) return cudaErrorInvalidValue;
    const dim3 grid((16 * a.g.h + 127) / 128 * (a.both ? 2 : 1)), block(128);
#define QCD_DSF16(E, RD)                                         \
    if (a.epi == E && a.reduce == RD) {                          \
        dslash_fix16_kernel<E, RD><<<grid, block, 0, s>>>(a);    \
        return cudaGetLastError();                               \
    }
    QCD_DSF16(EPI_PLAIN, false)
    QCD_DSF16(EPI_CPLX_D, false)
    QCD_DSF16(EPI_REAL_YD, false)
    QCD_DSF16(EPI_REAL_YD, true)
    QCD_DSF16(EPI_CPLX_YD, false)
    QCD_DSF16(EPI_CPLX_YD, true)
#undef QCD_DSF16
    return cudaErrorInvalidValue;
}

template <int D>
cudaError_t launch_dslash_fix_multi(const DslashMulti &a, cudaStream_t s)
{
    const dim3 grid((unsigned)((a.g.h + kFixElems - 1) / kFixElems) * a.n * (a.both ? 2 : 1)), block(kFixThreads);
    dslash_fix_kernel<D, EPI_PLAIN, false, DslashMulti><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

template <int D>
cudaError_t launch_dslash_fix_dag(const DslashLaunch &a, cudaStream_t s)
{
    const dim3 grid((((a.g.h << a.rhs_log2) + kFixElems - 1) / kFixElems) * (a.both ? 2 : 1)), block(kFixThreads);
#define QCD_DSF(E, RD)                                               \
    if (a.epi == E && a.reduce == RD) {                              \
        dslash_fix_kernel<D, E, RD><<<grid, block, 0, s>>>(a);       \
        return cudaGetLastError();                                   \
    }
    QCD_DSF(EPI_PLAIN, false)
    QCD_DSF(EPI_CPLX_D, false)
    QCD_DSF(EPI_REAL_YD, false)
    QCD_DSF(EPI_REAL_YD, true)
    QCD_DSF(EPI_CPLX_YD, false)
    QCD_DSF(EPI_CPLX_YD, true)
#undef QCD_DSF
    return cudaErrorInvalidValue;
}

}  // namespace qcd
