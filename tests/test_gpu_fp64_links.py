"""The FP64 and double-float arithmetic kernels, which links outside the
fixed-point form take (csrc/fixed.cuh): SU(3) links times four, so that
entries exceed 1, against the FP64 oracle on the same links.

M depends on kappa U only, so kappa / 4 makes it the matrix of the SU(3) links,
exactly (powers of two): the solves converge as theirs do.  Threads per site:
0 the autotuner's choice, 1 one thread, 8 the lane kernel.  Bounds: D adds 24
products of each component's eight neighbours, in FP64 on both sides, so the
2-norm errors stay below a few 2^-53 of the result; double-float a few 2^-48.
"""

import numpy as np
import pytest

import oracle
from paper_1411_5219_gb300 import synthetic as syn
from tests import _fields as F
from tests._solves import schur_residual_oracle

pytestmark = pytest.mark.gpu

SCALE = 4.0


@pytest.fixture(scope="module")
def q():
    from paper_1411_5219_gb300 import _build, qcd
    _build.build()
    import torch
    assert torch.cuda.is_available()
    return qcd


@pytest.fixture(params=[0, 1, 8])
def threads(q, request):
    q.set_hop_threads(request.param)
    yield request.param
    q.set_hop_threads(0)


def _gauge(q, dims, seed=2001, t_bc=-1):
    lat = q.Lattice(dims, t_bc)
    U = SCALE * syn.gauge_field(dims, 0.2, seed)
    g = q.Gauge(lat, "f64", 18)
    g.upload(U)
    return lat, U, g


# less than a block, ragged tails, many blocks
DIMS = [(2, 2, 2, 2), (6, 4, 2, 8), (12, 10, 8, 6)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-15), ("df64", 1e-13)])
def test_dslash(q, threads, dims, dagger, prec, tol):
    lat, U, g = _gauge(q, dims, t_bc=1 if dagger else -1)
    bc = lat.t_bc
    psi = syn.gaussian_spinor(dims, 2002)
    for p in (0, 1):
        i, o = (q.Spinor(lat, ("even", "odd")[k], prec) for k in (1 - p, p))
        i.upload(syn.to_half(psi, 1 - p))
        q.apply_dslash(g, o, i, dagger=dagger)
        assert F.rel_err(o.download(), oracle.dhop_eo(U, syn.to_half(psi, 1 - p), p, t_bc=bc, dagger=dagger)) < tol
    i, o = q.Spinor(lat, "full", prec), q.Spinor(lat, "full", prec)
    i.upload(psi)
    q.apply_dslash(g, o, i, dagger=dagger)
    assert F.rel_err(o.download(), oracle.dhop(U, psi, t_bc=bc, dagger=dagger)) < tol


@pytest.mark.parametrize("mu", [0.0, 0.4])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-15), ("df64", 1e-13)])
def test_matrix(q, threads, mu, dagger, prec, tol):
    dims, kappa = (6, 4, 2, 8), 0.15 / SCALE
    mu *= SCALE  # (a = 2 kappa mu as for the SU(3) links)
    lat, U, g = _gauge(q, dims)
    psi = syn.gaussian_spinor(dims, 2003)
    i, o = q.Spinor(lat, "full", prec), q.Spinor(lat, "full", prec)
    i.upload(psi)
    q.apply_M(g, o, i, kappa, mu, eo=False, dagger=dagger)
    assert F.rel_err(o.download(), oracle.apply_m(U, psi, kappa, mu, dagger=dagger)) < tol
    i, o = q.Spinor(lat, "even", prec), q.Spinor(lat, "even", prec)
    i.upload(syn.to_half(psi, 0))
    q.apply_M(g, o, i, kappa, mu, eo=True, dagger=dagger)
    assert F.rel_err(o.download(), oracle.apply_mhat(U, syn.to_half(psi, 0), kappa, mu, dagger=dagger)) < tol


@pytest.mark.parametrize("nrhs", [1, 5, 32])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-15), ("df64", 1e-13)])
def test_multi(q, nrhs, prec, tol):
    dims = (6, 2, 4, 10)
    lat, U, g = _gauge(q, dims)
    psi = [syn.gaussian_spinor(dims, 2010 + k) for k in range(nrhs)]
    ins, outs = ([q.Spinor(lat, "full", prec) for _ in psi] for _ in range(2))
    for s, v in zip(ins, psi):
        s.upload(v)
    q.apply_dslash_multi(g, outs, ins)
    for k, v in enumerate(psi):
        assert F.rel_err(outs[k].download(), oracle.dhop(U, v)) < tol, k


@pytest.mark.parametrize("inner", ["f64", "f16", "df64"])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("eo", [True, False])
def test_solve(q, threads, inner, nrhs, eo):
    """With mu the complex epilogues, without it the real ones; the fused norm
    in FP64 and the FP64 defect and verification of the mixed solver."""
    dims = (4, 6, 4, 4)
    lat, U, g = _gauge(q, dims)
    for mu in (0.0, 0.02):
        kappa, src = 0.14 / SCALE, [syn.gaussian_spinor(dims, 2050 + k) for k in range(nrhs)]
        b, x = ([q.Spinor(lat, "full", "f64") for _ in src] for _ in range(2))
        for s, v in zip(b, src):
            s.upload(v)
        status, stats = q.solve_cg_multi(g, x, b, kappa, mu * SCALE, tol=1e-11, eo=eo, inner_prec=inner, inner_recon=18)
        assert status == 0
        for k, v in enumerate(src):
            assert stats[k]["true_rel_residual"] <= 1e-11
            want, _ = oracle.solve_eo(U, v, kappa, mu * SCALE, tol=1e-13)
            assert F.rel_err(x[k].download(), want) < 1e-9


def test_many(q):
    """The eight-lane FP64 phases of the persistent solver, beside a system in
    fixed point."""
    probs = []
    for dims, seed, scale in (((4, 4, 4, 4), 2071, SCALE), ((6, 4, 4, 8), 2072, SCALE), ((6, 4, 2, 8), 2073, 1.0)):
        lat = q.Lattice(dims, -1)
        U = scale * syn.gauge_field(dims, 0.2, seed)
        g = q.Gauge(lat, "f64", 18)
        g.upload(U)
        v = syn.gaussian_spinor(dims, seed + 10)
        b, x = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
        b.upload(v)
        probs.append((g, x, b, 0.14 / scale, 0.02 * scale, U, v))
    g, x, b, kappa, mu, Us, vs = zip(*probs)
    status, stats = q.solve_cg_many(g, x, b, kappa, mu, [1e-11] * 3)
    assert status == 0
    for k in range(3):
        assert stats[k]["true_rel_residual"] <= 1e-11
        assert schur_residual_oracle(Us[k], vs[k], x[k].download(), kappa[k], mu[k]) <= 1.5e-11


@pytest.mark.parametrize("first,then", [(1, 8), (8, 1)])
def test_solve_takes_the_shape_set_last(q, first, then):
    """A solve after qcd_set_hop_threads does not replay the graph of one before
    it: the bits are those of a lattice that only knows the later setting."""
    dims = (6, 4, 2, 8)
    b = syn.gaussian_spinor(dims, 2091)
    out = []
    try:
        for settings in ((first, then), (then,)):
            lat, U, g = _gauge(q, dims, seed=2090)
            bs, x = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
            bs.upload(b)
            for tps in settings:
                q.set_hop_threads(tps)
                q.solve_cg(g, x, bs, 0.14 / SCALE, 0.02 * SCALE)
            out.append(x.download())
    finally:
        q.set_hop_threads(0)
    assert np.array_equal(out[0], out[1])
