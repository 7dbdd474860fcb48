// The FP64 hopping term in integer arithmetic: formats and the hop.
//
// GB300 starts one FP64 warp instruction per sub-partition every 64 cycles,
// so the ~790 of a site cost a warp 51,000 cycles however fast its data
// arrives: 48^3 x 12 took 945 us for bytes that HBM moves in 151 us.  The
// same SU(3) products in 60-bit fixed point are 32 x 32 + 64 bit integer
// multiply-adds, many times cheaper.  The operation is the Wilson hop of
// CL2QCD (arXiv:1411.5219, Sec. 1 and 6), in the chiral basis of
// dslash_kernel.cuh.
//
//   Links (int4 per complex entry, the bytes of the FP64 form): entries of
//     magnitude <= 1 as V = round(u 2^60) = vh 2^30 + vl, |vl| <= 2^29.
//   Spinors (SpFix: int4 per complex component and one exponent E per site):
//     P = trunc(psi 2^(1078 - E)) = ph 2^30 + pl, |pl| <= 2^29, with E the
//     largest FP64 exponent field of the site's 24 reals: |P| < 2^56.
//   Projection: limb by limb, no carries (|ph| <= 2^27, -2^30 <= pl < 2^30).
//   Products: ph vh at weight 2^60 and ph vl + pl vh at weight 2^30, summed
//     exactly over the six real products of an entry (below 2^63); pl vl, about
//     half a unit of P, is left out.  Gauss's three products for a complex one:
//     his intermediate sums may wrap, the final ones do not.
//   Sums over the eight hops: exact in 64 bits (below 48 * 2^57) once shifted to
//     the largest E of the eight neighbours.
//
// Errors, in units of P of the largest neighbour (2^-55 of its largest real at
// most), for one real of one hop with SU(3) links: below 2 for each real of the
// half spinor (psi is truncated), times at most sqrt(6) for the row of U, 4.9;
// 3 for the low products; 0.4 for the links' rounding; 0.5 and 1 for the two
// shifts.  Below 10 a hop, 2^-48 of the largest real over eight; measured at
// 12^3 x 6 2^-50.6 (FP64 arithmetic 2^-49.2).  In the 2-norm (against 128-bit
// arithmetic) 5e-17 of the result on Gaussian fields, 1.6e-16 in FP64, and the
// median component is closer too (2^-54 of its own size, 2^-53).  Not so a
// component far below the others of its sites that the links do not mix with
// them: it has the bits above 2^-55 of the largest.  With components spread over
// 10^-12 .. 1: 1.2e-16 and 1.5e-16 in the 2-norm, the worst component 2^-42 and
// 2^-46 of its own size; with unit links 1.1e-16 and 1.0e-16, 2^-34 and 2^-47.
//
// Sites that fixed point does not hold -- a non-finite component, or a largest
// exponent near either end of the range -- keep their FP64 values (E =
// kFixRaw), and the sites next to them are computed in FP64.
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

using i64 = long long;

constexpr int kPrecFix = 5;     // storage of internal fields next to qcd_prec
constexpr int kFixRadix = 30;   // bits of the low limbs
constexpr int kFixBits = 56;    // |P| < 2^56
constexpr int kFixBias = 1078;  // value = P 2^(E - kFixBias)
constexpr int kFixRaw = 4095;   // exponent of a site stored as FP64
constexpr int kFixLow = 128, kFixHigh = 1980;  // exponent fields outside are stored as FP64

// (sums wrap: an intermediate one may leave the range that the final one keeps)
__device__ __forceinline__ i64 wadd(i64 a, i64 b) { return (i64)((unsigned long long)a + (unsigned long long)b); }
__device__ __forceinline__ i64 wsub(i64 a, i64 b) { return (i64)((unsigned long long)a - (unsigned long long)b); }
__device__ __forceinline__ i64 madw(int a, int b, i64 c) { return wadd((i64)a * (i64)b, c); }

// P in limbs.
__device__ __forceinline__ void to_limbs(i64 P, int &hi, int &lo)
{
    hi = (int)((P + (1ll << (kFixRadix - 1))) >> kFixRadix);
    lo = (int)P - (hi << kFixRadix);
}
__device__ __forceinline__ i64 of_limbs(int hi, int lo) { return madw(hi, 1 << kFixRadix, lo); }

// The high word without its sign: orders magnitudes, the exponent field on top.
__device__ __forceinline__ unsigned twice_hi(double v) { return (unsigned)__double2hiint(v) << 1; }

// P of one real at exponent field E >= its own (a zero of a site with E >= 128
// shifts to nothing).
__device__ __forceinline__ i64 fix_of(double v, int E)
{
    const int H = __double2hiint(v);
    const unsigned L = (unsigned)__double2loint(v);
    const int d = E - (int)(((unsigned)H << 1) >> 21);
    const unsigned mh = ((unsigned)H & 0x000fffffu) | 0x00100000u;
    const unsigned long long m = ((unsigned long long)__funnelshift_l(L, mh, 3) << 32) | (L << 3);
    const i64 P = (i64)(m >> min(d, 63));
    return H < 0 ? -P : P;
}

// P 2^(E - kFixBias) as a double (rounded to 53 bits).
__device__ __forceinline__ double fix_value(i64 P, int E)
{
    const double v = __ll2double_rn(P);
    const int hi = __double2hiint(v) + ((E - kFixBias) << 20);
    return P != 0 ? __hiloint2double(hi, __double2loint(v)) : 0.0;
}

// The same for a P of at most 53 significant bits (one that came from a
// double), exactly and without FP64 instructions: a 64-bit conversion holds
// the FP64 pipe for 74 cycles a warp, these dozen integer instructions do not.
__device__ __forceinline__ double fix_value_exact(i64 P, int E)
{
    const unsigned long long m = (unsigned long long)(P < 0 ? -P : P);
    const int z = __clzll((long long)m);
    const unsigned long long n = m << (z & 63);  // leading one at bit 63
    // (the leading one adds one to the exponent field)
    const int hi = ((E - kFixBias + 1023 + 62 - z) << 20) + (int)(n >> 43);
    const int lo = (int)(n >> 11);
    return P == 0 ? 0.0 : __hiloint2double(hi | (P < 0 ? (int)0x80000000 : 0), lo);
}

// The exponent that a site is stored under: `top` its largest twice_hi, `low`
// an or of its low words (wanted where top is zero: the smallest denormals).
__device__ __forceinline__ int fix_exponent(unsigned top, unsigned low)
{
    const int E = (int)(top >> 21);
    return (top | low) == 0u ? 0 : (E < kFixLow || E > kFixHigh) ? kFixRaw : E;
}

// One stored component as FP64 (what the hop itself wrote may hold 56 bits:
// cut to 53 here).
__device__ __forceinline__ double2 fix_load(int4 q, int E)
{
    if (E == kFixRaw) return make_double2(__hiloint2double(q.y, q.x), __hiloint2double(q.w, q.z));
    return make_double2(fix_value_exact(of_limbs(q.x, q.y), E), fix_value_exact(of_limbs(q.z, q.w), E));
}
__device__ __forceinline__ int4 fix_store(double re, double im, int E)
{
    int4 q;
    if (E == kFixRaw) {
        q = make_int4(__double2loint(re), __double2hiint(re), __double2loint(im), __double2hiint(im));
    } else if (E == 0) {
        q = make_int4(0, 0, 0, 0);
    } else {
        to_limbs(fix_of(re, E), q.x, q.y);
        to_limbs(fix_of(im, E), q.z, q.w);
    }
    return q;
}

// A fixed-point half field for the site kernels: FP64 in and out.  The
// exponents lie where FP16 fields keep their scales.
struct SpFix {
    using R = double;
    static constexpr int kPlanes = 12;
    static constexpr size_t kBytesPerSite = 196;
    static constexpr bool kScaled = false;
    __device__ __forceinline__ static int exponent(const SpinorView &v, int i)
    {
        return __ldg(reinterpret_cast<const int *>(v.norm) + i);
    }
    __device__ __forceinline__ static Spinor<R> load(const SpinorView &v, int i)
    {
        Spinor<R> s;
        const int4 *p = static_cast<const int4 *>(v.data) + i;
        const int E = exponent(v, i);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const double2 d = fix_load(__ldg(p + (size_t)k * v.stride), E);
            s.c[k / 3][k % 3] = mk(d.x, d.y);
        }
        return s;
    }
    __device__ __forceinline__ static void store(const SpinorView &v, int i, const Spinor<R> &s)
    {
        unsigned top = 0u, low = 0u;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const cx<R> v2 = s.c[k / 3][k % 3];
            top = max(top, max(twice_hi(v2.re), twice_hi(v2.im)));
            low |= (unsigned)(__double2loint(v2.re) | __double2loint(v2.im));
        }
        const int E = fix_exponent(top, low);
        int4 *p = static_cast<int4 *>(v.data) + i;
#pragma unroll
        for (int k = 0; k < 12; ++k) p[(size_t)k * v.stride] = fix_store(s.c[k / 3][k % 3].re, s.c[k / 3][k % 3].im, E);
        reinterpret_cast<int *>(v.norm)[i] = E;
    }
};

// The epilogue cy y + cd v of one complex component: fewer FP64 instructions
// where cy is 1 or 1 + i a and cd real, as in M and its Schur complement.
template <bool kReal>
__device__ __forceinline__ cx<double> fix_epilogue(cx<double> v, double2 y, cx<double> cy, cx<double> cd)
{
    if (kReal) {
        if (cy.re == 1.0) return mk(fma(cd.re, v.re, y.x), fma(cd.re, v.im, y.y));
        return mk(fma(cd.re, v.re, cy.re * y.x), fma(cd.re, v.im, cy.re * y.y));
    }
    if (cy.re == 1.0 && cd.im == 0.0)
        return mk(fma(cd.re, v.re, fma(-cy.im, y.y, y.x)), fma(cd.re, v.im, fma(cy.im, y.x, y.y)));
    return cmac(cmul(cy, mk(y.x, y.y)), cd, v);
}

// The sums of one thread: spin s of the output (up) and what its spin s of
// the half spinors gives to the lower spins, 2 + s in the z and t hops (la),
// 3 - s in the x and y hops (lb): re, im of three colours.
struct FixAcc {
    i64 up[6], la[6], lb[6];
};

__device__ __forceinline__ void negate_all(i64 (&v)[6], bool neg)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = neg ? -v[k] : v[k];
}

// One hop of one spin: project, multiply and accumulate.  sg: +-1 on the
// second spin's term, where it depends on s (y and z hops); shift: to the
// exponent of the sums.  kStage: which sums hold something already (order y,
// x, z, t: 0 none, 1 up and lb, 2 all).  The lower spins of y and z are
// negated by the caller for s = 1.  a, b: psi of spin s and of the spin that
// it is projected with (components kSites apart), u: the link (entries
// kSites apart), all in shared memory.
template <int MU, int S, bool kAdj, int kStage, int kSites>
__device__ __forceinline__ void hop_fix(FixAcc &acc, const int4 *pa, const int4 *pb, const int4 *u, int sg, int shift,
                                        bool flip)
{
    constexpr int w = MU == 3 ? -S : S;
    int fh[6], fl[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int4 a = pa[c * kSites], b = pb[c * kSites];
        // (limbs of b's parts in the order they meet a's, without their signs)
        const int xh = (MU == 0 || MU == 2) ? b.z : b.x, xl = (MU == 0 || MU == 2) ? b.w : b.y;
        const int yh = (MU == 0 || MU == 2) ? b.x : b.z, yl = (MU == 0 || MU == 2) ? b.y : b.w;
        constexpr int wr = (MU == 0 || MU == 2) ? -w : w;  // i b = (-im, re)
        if (MU == 1 || MU == 2) {
            fh[2 * c] = a.x + wr * sg * xh;
            fl[2 * c] = a.y + wr * sg * xl;
            fh[2 * c + 1] = a.z + w * sg * yh;
            fl[2 * c + 1] = a.w + w * sg * yl;
        } else {
            fh[2 * c] = a.x + wr * xh;
            fl[2 * c] = a.y + wr * xl;
            fh[2 * c + 1] = a.z + w * yh;
            fl[2 * c + 1] = a.w + w * yl;
        }
    }
    // Gauss's three products of a complex one: with P1 = ur (hr + hi),
    // P2 = (ui - ur) hr and P3 = (ur + ui) hi, U h = (P1 - P3) + i (P1 + P2);
    // conj(U) h = (P1 + (ui - ur) hi) + i (P1 - (ur + ui) hr)
    int sh[3], sl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        sh[c] = fh[2 * c] + fh[2 * c + 1];
        sl[c] = fl[2 * c] + fl[2 * c + 1];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // (the half unit of weight 2^30 rounds the shift below)
        i64 h1 = 0, m1 = 1ll << (kFixRadix - 1), h2 = 0, m2 = 0, h3 = 0, m3 = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 v = u[(kAdj ? 3 * b + a : 3 * a + b) * kSites];  // re hi, re lo, im hi, im lo
            const int xh = v.x + v.z, xl = v.y + v.w, yh = v.z - v.x, yl = v.w - v.y;
            // the factors of ui - ur and ur + ui
            const int dh = fh[2 * b + (kAdj ? 1 : 0)], dl = fl[2 * b + (kAdj ? 1 : 0)];
            const int eh = fh[2 * b + (kAdj ? 0 : 1)], el = fl[2 * b + (kAdj ? 0 : 1)];
            h1 = madw(v.x, sh[b], h1);
            m1 = madw(v.x, sl[b], m1);
            m1 = madw(v.y, sh[b], m1);
            h2 = madw(yh, dh, h2);
            m2 = madw(yh, dl, m2);
            m2 = madw(yl, dh, m2);
            h3 = madw(xh, eh, h3);
            m3 = madw(xh, el, m3);
            m3 = madw(xl, eh, m3);
        }
        const i64 plus = wadd(h1, h2) + (wadd(m1, m2) >> kFixRadix), minus = wsub(h1, h3) + (wsub(m1, m3) >> kFixRadix);
        i64 ur = (kAdj ? plus : minus) >> shift, ui = (kAdj ? minus : plus) >> shift;
        if (flip) {
            ur = -ur;
            ui = -ui;
        }
        // the lower spin: x, z: -S i u; y: +S u; t: -S u
        i64 lr, li;
        if (MU == 0 || MU == 2) {
            lr = S > 0 ? ui : -ui;
            li = S > 0 ? -ur : ur;
        } else {
            constexpr bool neg = (MU == 1) != (S > 0);
            lr = neg ? -ur : ur;
            li = neg ? -ui : ui;
        }
        acc.up[2 * a] = kStage == 0 ? ur : acc.up[2 * a] + ur;
        acc.up[2 * a + 1] = kStage == 0 ? ui : acc.up[2 * a + 1] + ui;
        if (MU <= 1) {
            acc.lb[2 * a] = kStage == 0 ? lr : acc.lb[2 * a] + lr;
            acc.lb[2 * a + 1] = kStage == 0 ? li : acc.lb[2 * a + 1] + li;
        } else {
            acc.la[2 * a] = kStage == 1 ? lr : acc.la[2 * a] + lr;
            acc.la[2 * a + 1] = kStage == 1 ? li : acc.la[2 * a + 1] + li;
        }
    }
}

}  // namespace qcd
