"""The fixed-point FP64 hopping kernels (csrc/fixed.cuh, csrc/fix_lanes.cuh)
against the FP64 oracle.

qcd_set_hop_threads forces the thread pair per element (1) and the sixteen
lanes (8) whatever the lattice.  Bounds: norm-wise 1e-15, a few 2^-53 of the
oracle's own; real by real ten units of 2^-55 of the largest real a hop, 2^-48 of
the largest over the eight neighbours (csrc/fixed.cuh; the oracle adds about 2^-50).
"""

import numpy as np
import pytest

import oracle
from paper_1411_5219_gb300 import synthetic as syn
from tests import _fields as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    from paper_1411_5219_gb300 import _build, qcd
    _build.build()
    import torch
    assert torch.cuda.is_available()
    return qcd


@pytest.fixture(autouse=True, params=[1, 8])
def threads(q, request):
    q.set_hop_threads(request.param)
    yield
    q.set_hop_threads(0)


def _gauge(q, dims, seed=1501, scale=1.0):
    lat = q.Lattice(dims, -1)
    U = scale * syn.gauge_field(dims, 0.3, seed)
    g = q.Gauge(lat, "f64", 18)
    g.upload(U)
    return lat, U, g


def _apply(q, lat, g, psi, out_par, dagger=False):
    si, so = (q.Spinor(lat, ("even", "odd")[p], "f64") for p in (1 - out_par, out_par))
    si.upload(syn.to_half(psi, 1 - out_par))
    q.apply_dslash(g, so, si, dagger=dagger)
    return so.download()


# less than a warp, one element over a block of 64, ragged tails, many blocks
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 4, 2), (10, 2, 2, 6), (4, 6, 10, 2), (12, 10, 8, 6)])
@pytest.mark.parametrize("dagger", [False, True])
def test_fixed_dslash(q, dims, dagger):
    lat, U, g = _gauge(q, dims)
    psi = syn.gaussian_spinor(dims, 1502)
    for p in (0, 1):
        want = oracle.dhop_eo(U, syn.to_half(psi, 1 - p), p, dagger=dagger)
        assert F.rel_err(_apply(q, lat, g, psi, p, dagger), want) < 1e-15


def _neighbour_max(psi):
    """Per site the sum of the largest |real component| of the eight neighbours."""
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-2, -1))
    return sum(np.roll(m, s, a) for a in range(4) for s in (1, -1))


@pytest.mark.parametrize("case", ["range", "extreme", "nonfinite", "zeros"])
def test_fixed_unusual_values(q, case):
    """Sites far apart in magnitude, beyond the range of the fixed form (largest
    exponents, denormals), infinities and NaN, and exact zeros."""
    dims = (8, 6, 4, 6)
    lat, U, g = _gauge(q, dims)
    psi = syn.gaussian_spinor(dims, 1503)
    flat = psi.reshape(-1, 12)
    rng = np.random.default_rng(5)
    if case == "range":
        flat *= 10.0 ** rng.uniform(-200, 200, (len(flat), 1))
        flat *= 10.0 ** rng.uniform(-12, 0, flat.shape)
    elif case == "extreme":
        for k, f in enumerate((1e300, 1e-300, 1e-310, 4e-324, 1e290, 1e-270)):
            flat[k::37] = flat[k::37] * f if f != 4e-324 else f
    elif case == "nonfinite":
        flat[5, 3] = np.nan
        flat[40, 0] = np.inf
        flat[77, 11] = -np.inf * 1j
    else:
        flat[:] = np.where(rng.random(flat.shape) < 0.97, 0.0, flat)
        flat[:5] = -0.0
    for p in (0, 1):
        got = _apply(q, lat, g, psi, p)
        with np.errstate(all="ignore"):
            want = oracle.dhop_eo(U, syn.to_half(psi, 1 - p), p)
            bound = syn.to_half(np.broadcast_to(_neighbour_max(psi)[..., None, None], psi.shape).copy(), p)
            fine = np.isfinite(want).all(axis=(1, 2))
            assert np.array_equal(fine, np.isfinite(got).all(axis=(1, 2)))
            assert np.all(np.abs(got - want)[fine] <= 1e-15 * bound[fine] + 1e-322)
        if case == "zeros":
            assert np.all(got[bound[:, 0, 0] == 0] == 0)


@pytest.mark.parametrize("links", ["su3", "near unit", "unit", "diagonal"])
@pytest.mark.parametrize("spread", [0, 3, 12])
def test_component_bound(q, links, spread):
    """The stated bound of each real, with components of a site spread over
    orders of magnitude and links that keep them apart."""
    dims = (8, 6, 4, 6)
    lat = q.Lattice(dims, -1)
    U = syn.gauge_field(dims, 0.01 if links == "near unit" else 0.3, 1551)
    rng = np.random.default_rng(1552)
    if links in ("unit", "diagonal"):
        phase = np.zeros(U.shape[:-1]) if links == "unit" else rng.uniform(-np.pi, np.pi, U.shape[:-1])
        phase[..., 2] = -phase[..., 0] - phase[..., 1]
        U = np.exp(1j * phase)[..., None] * np.eye(3)
    g = q.Gauge(lat, "f64", 18)
    g.upload(U)
    psi = syn.gaussian_spinor(dims, 1553)
    psi *= 10.0 ** rng.uniform(-spread, 0, psi.shape)
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-2, -1))
    m = np.max([np.roll(m, s, a) for a in range(4) for s in (1, -1)], axis=0)
    for p in (0, 1):
        d = _apply(q, lat, g, psi, p) - oracle.dhop_eo(U, syn.to_half(psi, 1 - p), p)
        bound = syn.to_half(np.broadcast_to(m[..., None, None], psi.shape).astype(complex), p).real
        assert np.all(np.maximum(np.abs(d.real), np.abs(d.imag)) <= (2.0 ** -48 + 2.0 ** -50) * bound)


def test_links_beyond_the_fixed_form_stay_fp64(q):
    """Entries above 1 take the FP64 kernels; the next upload is looked at again."""
    dims = (6, 4, 4, 4)
    lat, U, g = _gauge(q, dims, scale=3.0)
    psi = syn.gaussian_spinor(dims, 1504)
    want = oracle.dhop_eo(U, syn.to_half(psi, 1), 0)
    assert F.rel_err(_apply(q, lat, g, psi, 0), want) < 1e-14
    g.upload(U / 3.0)
    assert F.rel_err(3.0 * _apply(q, lat, g, psi, 0), want) < 2e-15


def test_first_use_under_stream_capture(q):
    """Without the fixed-point copies yet, a captured launch is the FP64 kernel."""
    import torch
    dims = (6, 4, 4, 4)
    lat, U, g = _gauge(q, dims)
    psi = syn.gaussian_spinor(dims, 1505)
    si, so = q.Spinor(lat, "odd", "f64"), q.Spinor(lat, "even", "f64")
    si.upload(syn.to_half(psi, 1))
    q.stream_sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        q.apply_dslash(g, so, si)
    graph.replay()
    torch.cuda.synchronize()
    assert F.rel_err(so.download(), oracle.dhop_eo(U, syn.to_half(psi, 1), 0)) < 1e-15


@pytest.mark.parametrize("mu", [0.0, 0.02])
@pytest.mark.parametrize("nrhs", [1, 17])
@pytest.mark.parametrize("eo", [True, False])
def test_fixed_solves(q, mu, nrhs, eo):
    """FP64 CG with its operator fields in fixed point, alone and as a batch of
    32 (17 and its padding: two elements of a right-hand side per warp)."""
    dims, kappa = (4, 6, 4, 4), 0.14
    lat, U, g = _gauge(q, dims)
    src = [syn.gaussian_spinor(dims, 1510 + k) for k in range(nrhs)]
    bs, xs = [q.Spinor(lat, "full", "f64") for _ in src], [q.Spinor(lat, "full", "f64") for _ in src]
    for b, s in zip(bs, src):
        b.upload(s)
    _, stats = q.solve_cg_multi(g, xs, bs, kappa, mu, tol=1e-11, eo=eo)
    for k in range(0, nrhs, 8):
        assert stats[k]["true_rel_residual"] <= 1e-11
        want, _ = oracle.solve_eo(U, src[k], kappa, mu, tol=1e-13)
        assert F.rel_err(xs[k].download(), want) < 1e-9


@pytest.mark.parametrize("inner,per_update", [("f64", 1), ("f16", 2)])
def test_launch_count_of_a_solve_holds_the_conversions(q, inner, per_update):
    """The thread pairs convert FP64 inputs in launches of their own, the lanes do
    not: three outside the loop (source, odd sites, residual), and per reliable
    update x and, in mixed precision, the defect."""
    dims = (4, 6, 4, 4)
    lat, U, g = _gauge(q, dims)
    b, x = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
    b.upload(syn.gaussian_spinor(dims, 1520))
    count = {}
    for tps in (8, 1):
        q.set_hop_threads(tps)
        for _ in range(2):  # (the first solve builds its graph)
            n0 = q.kernel_launches()
            _, st = q.solve_cg(g, x, b, 0.14, 0.02, tol=1e-10, inner_prec=inner)
            count[tps] = q.kernel_launches() - n0, st["iterations"], st["reliable_updates"]
    assert count[1][1:] == count[8][1:]
    assert count[1][0] - count[8][0] == 3 + per_update * count[1][2]
