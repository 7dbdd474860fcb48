"""Calls that find no memory for a workspace (the allocation fails by injection
on the host): they give back what the fixed-point form of the FP64 operators
took and run in FP64 arithmetic, with the oracle's result."""

import pytest

import oracle
from paper_1411_5219_gb300 import synthetic as syn
from tests import _fields as F

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 2, 8)
KAPPA, MU = 0.14, 0.02


@pytest.fixture(scope="module")
def q():
    from paper_1411_5219_gb300 import _build, qcd
    _build.build()
    import torch
    assert torch.cuda.is_available()
    return qcd


@pytest.fixture(autouse=True)
def threads(q):
    q.set_hop_threads(1)
    yield
    q.debug_inject(q.INJECT_WORKSPACE, 0)
    q.set_hop_threads(0)


def _setup(q, seed):
    lat = q.Lattice(DIMS, -1)
    U = syn.gauge_field(DIMS, 0.3, seed)
    g = q.Gauge(lat, "f64", 18)
    g.upload(U)
    psi = syn.gaussian_spinor(DIMS, seed + 1)
    i, o = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
    i.upload(psi)
    g.prepare("f64", 18)
    q.stream_sync()
    return lat, U, g, psi, i, o


def _half(q, lat, g, psi):
    e, r = q.Spinor(lat, "even", "f64"), q.Spinor(lat, "even", "f64")
    e.upload(syn.to_half(psi, 0))
    q.apply_M(g, r, e, KAPPA, MU, eo=True)
    return r.download()


def _solve(q, lat, g, psi, i, o, inner="f64"):
    status, st = q.solve_cg(g, o, i, KAPPA, MU, tol=1e-11, inner_prec=inner)
    assert status == 0 and st["true_rel_residual"] <= 1e-11
    return o.download()


def _many(q, lat, g, psi, i, o):
    status, _ = q.solve_cg_many([g], [o], [i], [KAPPA], [MU], [1e-11])
    assert status == 0
    return o.download()


def _multi(q, lat, g, psi, i, o):
    q.apply_dslash_multi(g, [o], [i])
    return o.download()


@pytest.mark.parametrize("what", ["mhat", "solve", "solve_f16", "many", "multi"])
def test_runs_without_memory_for_the_fixed_form(q, what):
    lat, U, g, psi, i, o = _setup(q, 1901)
    call = {"mhat": lambda: _half(q, lat, g, psi), "solve": lambda: _solve(q, lat, g, psi, i, o),
            "solve_f16": lambda: _solve(q, lat, g, psi, i, o, "f16"), "many": lambda: _many(q, lat, g, psi, i, o),
            "multi": lambda: _multi(q, lat, g, psi, i, o)}[what]
    if what == "mhat":
        want, tol = oracle.apply_mhat(U, syn.to_half(psi, 0), KAPPA, MU), 1e-15
    elif what == "multi":
        want, tol = oracle.dhop(U, psi), 1e-15
    else:
        want, tol = oracle.solve_eo(U, psi, KAPPA, MU, tol=1e-13)[0], 1e-9
    q.debug_inject(q.INJECT_WORKSPACE, 1)
    assert F.rel_err(call(), want) < tol
    for _ in range(2):  # in FP64 until an upload, then in fixed point again
        o.zero()
        assert F.rel_err(call(), want) < tol
        g.upload(U)


def test_a_copy_that_a_graph_holds_stays(q):
    """A caller's graph replays as before after a call that found no memory."""
    import torch
    lat, U, g, psi, i, o = _setup(q, 1911)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        q.apply_dslash(g, o, i)
    q.debug_inject(q.INJECT_WORKSPACE, 1)
    with pytest.raises(q.QcdError) as e:
        _half(q, lat, g, psi)
    assert e.value.status == 2  # QCD_ERR_OOM: nothing to give back
    q.debug_inject(q.INJECT_WORKSPACE, 0)
    o.zero()
    q.stream_sync()
    graph.replay()
    torch.cuda.synchronize()
    assert F.rel_err(o.download(), oracle.dhop(U, psi)) < 1e-15
