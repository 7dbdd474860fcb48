// The fixed-point hop (fixed.cuh) with sixteen threads per site: one hop and
// one spin of the half spinor each, FP64 fields in and out.
//
// For small lattices, where a thread's chain of instructions sets the time
// (the CG at 8^3 x 4: 1.29 ms, 1.93 ms with a thread pair per site, 1.85 ms
// with eight FP64 lanes; from 12^3 x 6 on the pairs win): a thread converts six
// of its neighbour's components (the exponent is the largest of the site's
// neighbourhood, so no sum needs a shift), does one colour vector's product and
// joins the sums by shuffles.
#pragma once

#include "fixed.cuh"
#include "hop_lanes.cuh"

namespace qcd {

// Components of an input half field: the double2 planes of an FP64 field
// (kCoherent: written earlier in the same kernel launch, read through L2), or
// a fixed-point field's elements of one right-hand side.
template <bool kCoherent>
struct PlaneLoad {
    const double2 *d;
    int stride;
    __device__ __forceinline__ double2 operator()(int plane, int nb) const
    {
        const double2 *q = d + (size_t)plane * stride + nb;
        return kCoherent ? __ldcg(q) : __ldg(q);
    }
};
struct FixLoad {
    SpinorView v;
    int rhs_log2, rhs;
    __device__ __forceinline__ double2 operator()(int plane, int nb) const
    {
        const int e = (nb << rhs_log2) | rhs;
        return fix_load(__ldg(static_cast<const int4 *>(v.data) + (size_t)plane * v.stride + e), SpFix::exponent(v, e));
    }
};

// D psi of one site in FP64, hop after hop (12 complex: 3 spin + colour): next
// to sites that fixed point does not hold.
template <typename Load>
static __device__ __noinline__ void hop_site_f64(const Geom &g, const int4 *fix, int us, const Load load, int p, int i,
                                                 bool dagger, double2 *out)
{
    for (int c = 0; c < 12; ++c) out[c] = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        cx<double> v[12];
        hop_lane(g,
                 [&](int plane, int li) {
                     const int4 q = __ldg(fix + (size_t)plane * us + li);
                     return make_double2(0x1p-60 * (double)of_limbs(q.x, q.y), 0x1p-60 * (double)of_limbs(q.z, q.w));
                 },
                 load, p, i, k, dagger, v);
        for (int c = 0; c < 12; ++c) {
            out[c].x += v[c].re;
            out[c].y += v[c].im;
        }
    }
}

__device__ __forceinline__ i64 negate_if(i64 v, bool n) { return n ? -v : v; }

// Lane l = 8 s + k of a site's sixteen: hop k = 2 mu + backward, spin s.  After
// the call, `E` is the exponent of the site's sums (kFixRaw: not computed) and
// the lanes with k & 3 < 3 hold in re, im colour k & 3 of spin s + 2 (k >> 2).
// fix: fixed-point links of stride us; load(plane, nb): component `plane` of
// the input at half-site nb.  Every lane of the warp must call it.
template <typename Load>
__device__ __forceinline__ void hop_fix16(const Geom &g, const int4 *fix, size_t us, const Load &load, int p, int i,
                                          int l, bool dagger, int &E, i64 &re, i64 &im)
{
    const SiteCoords c = site_coords(g, i, p);
    const int k = l & 7, mu = k >> 1;
    const bool s = l & 8, bwd = k & 1;
    int nb;
    bool flip = false;
    if (mu == 0) {
        const int xn = bwd ? (c.x == 0 ? g.L[0] - 1 : c.x - 1) : (c.x + 1 == g.L[0] ? 0 : c.x + 1);
        nb = i - c.xh + (xn >> 1);
    } else {
        const int L = g.L[mu], st = mu == 1 ? g.sy : mu == 2 ? g.sz : g.st, x = mu == 1 ? c.y : mu == 2 ? c.z : c.t;
        const bool wrap = bwd ? x == 0 : x == L - 1;
        nb = wrap ? (bwd ? i + (L - 1) * st : i - (L - 1) * st) : (bwd ? i - st : i + st);
        flip = mu == 3 && wrap && antiperiodic(g);
    }
    // psi of spin s and of the spin it is projected with
    const int pa = s ? 3 : 0, pb = 6 + (s != (mu <= 1) ? 3 : 0);
    double2 a[3], b[3];
    int4 v[3][3];  // rows of U (forward) or of its transpose
    const int4 *u = fix + (size_t)((bwd ? 1 - p : p) * 4 + mu) * 9 * us + (bwd ? nb : i);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        a[j] = load(pa + j, nb);
        b[j] = load(pb + j, nb);
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) v[j / 3][j % 3] = __ldg(u + (size_t)(bwd ? 3 * (j % 3) + j / 3 : j) * us);
    unsigned top = 0u, low = 0u;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        top = max(max(top, max(twice_hi(a[j].x), twice_hi(a[j].y))), max(twice_hi(b[j].x), twice_hi(b[j].y)));
        low |= (unsigned)(__double2loint(a[j].x) | __double2loint(a[j].y) | __double2loint(b[j].x) | __double2loint(b[j].y));
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        low |= __shfl_xor_sync(0xffffffffu, low, o);
    }
    E = fix_exponent(top, low);
    const int Ec = max(E, kFixLow);  // (all zero: any exponent will do)
    // h = psi_s + w psi_b or + w i psi_b; its conjugate for a backward hop,
    // whose product conj(U^T) h is the conjugate of U^T conj(h)
    const bool S = dagger == bwd, imag = !(mu & 1);                       // S: the projector sign is +
    const bool wneg = S == (mu == 3) ? true : false, odd = s && (mu == 1 || mu == 2);
    const bool w = wneg != odd;                                           // w < 0
    int fh[6], fl[6], sh[3], sl[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const i64 br = fix_of(b[j].x, Ec), bi = fix_of(b[j].y, Ec);
        const i64 hr = fix_of(a[j].x, Ec) + negate_if(imag ? -bi : br, w);
        const i64 hi = fix_of(a[j].y, Ec) + negate_if(imag ? br : bi, w);
        to_limbs(hr, fh[2 * j], fl[2 * j]);
        to_limbs(negate_if(hi, bwd), fh[2 * j + 1], fl[2 * j + 1]);
        sh[j] = fh[2 * j] + fh[2 * j + 1];
        sl[j] = fl[2 * j] + fl[2 * j + 1];
    }
    i64 up[6], lo[6];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        i64 h1 = 0, m1 = 1ll << (kFixRadix - 1), h2 = 0, m2 = 0, h3 = 0, m3 = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int4 q = v[r][j];
            const int xh = q.x + q.z, xl = q.y + q.w, yh = q.z - q.x, yl = q.w - q.y;
            h1 = madw(q.x, sh[j], h1);
            m1 = madw(q.x, sl[j], m1);
            m1 = madw(q.y, sh[j], m1);
            h2 = madw(yh, fh[2 * j], h2);
            m2 = madw(yh, fl[2 * j], m2);
            m2 = madw(yl, fh[2 * j], m2);
            h3 = madw(xh, fh[2 * j + 1], h3);
            m3 = madw(xh, fl[2 * j + 1], m3);
            m3 = madw(xl, fh[2 * j + 1], m3);
        }
        const i64 ur = negate_if(wsub(h1, h3) + (wsub(m1, m3) >> kFixRadix), flip);
        const i64 ui = negate_if(wadd(h1, h2) + (wadd(m1, m2) >> kFixRadix), flip != bwd);
        // the lower spin: x: -S i u; y: +S u, z: -S i u (negated for s = 1); t: -S u
        const bool n = (S != (mu == 1)) != odd;
        up[2 * r] = ur;
        up[2 * r + 1] = ui;
        lo[2 * r] = negate_if(imag ? -ui : ur, n);
        lo[2 * r + 1] = negate_if(imag ? ur : ui, n);
    }
    // x and y hops give to the lower spin of the other s; then the sums over
    // the hops, half of the lanes keeping the upper spin and half the lower
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const i64 o = __shfl_xor_sync(0xffffffffu, lo[j], 8);
        if (mu <= 1) lo[j] = o;
        const bool upper = !(k & 4);
        const i64 give = __shfl_xor_sync(0xffffffffu, upper ? lo[j] : up[j], 4);
        up[j] = (upper ? up[j] : lo[j]) + give;
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        up[j] += __shfl_xor_sync(0xffffffffu, up[j], 2);
        up[j] += __shfl_xor_sync(0xffffffffu, up[j], 1);
    }
    const int col = k & 3;
    re = col == 0 ? up[0] : col == 1 ? up[2] : up[4];
    im = col == 0 ? up[1] : col == 1 ? up[3] : up[5];
}

}  // namespace qcd
