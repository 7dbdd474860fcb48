"""Operator calls captured into a CUDA graph of the caller: a replay gives the
result of a call, whatever other calls on the lattice came between (against
the FP64 oracle).

qcd_set_hop_threads forces the thread pair per site (1), whose input goes
through a workspace of the lattice, and the sixteen lanes (8), on small
lattices.
"""

import numpy as np
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


@pytest.fixture(params=[1, 8])
def threads(q, request):
    q.set_hop_threads(request.param)
    yield request.param
    q.set_hop_threads(0)


def _setup(q, seed=1701):
    lat = q.Lattice(DIMS, -1)
    U = syn.gauge_field(DIMS, 0.3, seed)
    g = q.Gauge(lat, "f64", 18)
    g.upload(U)
    psi = syn.gaussian_spinor(DIMS, seed + 1)
    return lat, U, g, psi


class _Call:
    """One operator call on fields of its own: run() it, its result, the oracle's."""

    def __init__(self, q, lat, g, psi, kind, prec="f64", dagger=False):
        self.q, self.g, self.psi, self.kind, self.dagger = q, g, psi, kind, dagger
        p_in, p_out = {"half": ("odd", "even"), "mhat": ("even", "even")}.get(kind, ("full", "full"))
        self.i, self.o = q.Spinor(lat, p_in, prec), q.Spinor(lat, p_out, prec)
        self.i.upload({"half": lambda: syn.to_half(psi, 1), "mhat": lambda: syn.to_half(psi, 0)}.get(kind, lambda: psi)())

    def run(self):
        if self.kind in ("half", "full"):
            self.q.apply_dslash(self.g, self.o, self.i, dagger=self.dagger)
        else:
            self.q.apply_M(self.g, self.o, self.i, KAPPA, MU, eo=self.kind == "mhat", dagger=self.dagger)

    def error(self, U):
        got, d = self.o.download(), self.dagger
        if self.kind == "half":
            want = oracle.dhop_eo(U, syn.to_half(self.psi, 1), 0, dagger=d)
        elif self.kind == "full":
            want = oracle.dhop(U, self.psi, dagger=d)
        elif self.kind == "mhat":
            want = oracle.apply_mhat(U, syn.to_half(self.psi, 0), KAPPA, MU, dagger=d)
        else:
            want = oracle.apply_m(U, self.psi, KAPPA, MU, dagger=d)
        self.o.zero()
        return F.rel_err(got, want)


def _capture(q, run):
    import torch
    q.stream_sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    return graph


def _replay(graph):
    import torch
    graph.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("kind", ["half", "mhat"])
@pytest.mark.parametrize("larger", ["full", "m", "solve"])
def test_replay_after_a_larger_call(q, threads, kind, larger):
    """The workspaces that a captured launch holds are not replaced when a
    call on more of the lattice needs its own."""
    lat, U, g, psi = _setup(q)
    call = _Call(q, lat, g, psi, kind)
    call.run()
    graph = _capture(q, call.run)
    if larger == "solve":
        b, x = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
        b.upload(psi)
        q.solve_cg(g, x, b, KAPPA, MU, eo=False)
    else:
        _Call(q, lat, g, psi, larger).run()
    q.stream_sync()
    call.o.zero()
    _replay(graph)
    assert call.error(U) < 1e-15


@pytest.mark.parametrize("kind", ["half", "mhat", "full", "m"])
def test_capture_after_a_call_of_another_form(q, kind):
    """A call captured after one eager call needs no new workspace, whichever
    kernel the earlier call took."""
    lat, U, g, psi = _setup(q, seed=1711)
    call = _Call(q, lat, g, psi, kind, dagger=True)
    for first, then in ((8, 1), (1, 8)):
        q.set_hop_threads(first)
        call.run()
        q.set_hop_threads(then)
        try:
            graph = _capture(q, call.run)
        finally:
            q.set_hop_threads(0)
        call.o.zero()
        _replay(graph)
        assert call.error(U) < 1e-15


def test_double_float_replay(q):
    """A captured double-float operator holds no workspace that grows."""
    lat, U, g, psi = _setup(q, seed=1721)
    call = _Call(q, lat, g, psi, "half", prec="df64")
    call.run()
    graph = _capture(q, call.run)
    _Call(q, lat, g, psi, "full", prec="df64").run()
    q.stream_sync()
    call.o.zero()
    _replay(graph)
    assert call.error(U) < 1e-13


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("overlapping", [False, True])
def test_multi_capture_with_more_fields(q, threads, prec, overlapping):
    """apply_dslash_multi of eight fields captured after a call with five (or,
    gathered because an output is another one's input, with eight), replayed
    after one with sixteen and one on both halves."""
    lat, U, g, psi = _setup(q, seed=1731)
    fields = [syn.to_half(syn.gaussian_spinor(DIMS, 1740 + k), 1) for k in range(8)]
    full = [q.Spinor(lat, "full", prec) for _ in range(9)]
    ins, outs = ([q.Spinor(lat, p, prec) for _ in range(16)] for p in ("odd", "even"))
    for s, v in zip(ins, fields):
        s.upload(v)
    gathered = overlapping or prec == "df64"

    def call(n=8):
        if overlapping:  # both halves of field k + 1 from field k
            q.apply_dslash_multi(g, full[1:n + 1], full[:n])
        else:
            q.apply_dslash_multi(g, outs[:n], ins[:n])

    def fill():
        for k in range(8):
            full[k].upload(syn.gaussian_spinor(DIMS, 1740 + k))

    fill()
    call(8 if gathered else 5)
    graph = _capture(q, call)
    fill()
    q.apply_dslash_multi(g, outs, ins)
    q.apply_dslash_multi(g, [q.Spinor(lat, "full", prec) for _ in range(8)], full[:8])
    for o in outs:
        o.zero()
    q.stream_sync()
    _replay(graph)
    tol = 1e-15 if prec == "f64" else 1e-13
    for k in range(8):
        if overlapping:
            assert F.rel_err(full[k + 1].download(), oracle.dhop(U, syn.gaussian_spinor(DIMS, 1740 + k))) < tol, k
        else:
            assert F.rel_err(outs[k].download(), oracle.dhop_eo(U, fields[k], 0)) < tol, k


@pytest.mark.parametrize("kind", ["half", "full", "mhat", "m"])
@pytest.mark.parametrize("first", [1.0, 4.0])
def test_replay_after_uploads(q, threads, kind, first):
    """A replay applies the links of the last upload, also where those have
    entries above 1 (scaled by four), which the fixed-point form does not hold,
    and whatever eager calls came between."""
    lat, U, g, psi = _setup(q, seed=1751)
    g.upload(first * U)
    call = _Call(q, lat, g, psi, kind, dagger=True)
    call.run()
    graph = _capture(q, call.run)
    for k, (scale, eager) in enumerate([(1.0, False), (4.0, False), (4.0, True), (1.0, True), (1.0, False)]):
        V = scale * syn.gauge_field(DIMS, 0.3, 1760 + k)
        g.upload(V)
        if eager:
            call.run()
            assert call.error(V) < 1e-15, k
        q.stream_sync()
        _replay(graph)
        assert call.error(V) < 1e-15, k


def test_multi_replay_after_uploads(q, threads):
    lat, U, g, psi = _setup(q, seed=1771)
    fields = [syn.to_half(syn.gaussian_spinor(DIMS, 1780 + k), 1) for k in range(3)]
    ins, outs = ([q.Spinor(lat, p, "f64") for _ in fields] for p in ("odd", "even"))
    for s, v in zip(ins, fields):
        s.upload(v)
    q.apply_dslash(g, outs[0], ins[0])
    graph = _capture(q, lambda: q.apply_dslash_multi(g, outs, ins))
    for scale in (4.0, 1.0):
        V = scale * syn.gauge_field(DIMS, 0.3, 1772)
        g.upload(V)
        q.stream_sync()
        _replay(graph)
        for o, v in zip(outs, fields):
            assert F.rel_err(o.download(), oracle.dhop_eo(V, v, 0)) < 1e-15


def test_captured_upload(q, threads):
    """Replays of a captured upload change the links without a call of the
    library: eager operators and captured ones apply the new ones."""
    import torch
    lat, U, g, psi = _setup(q, seed=1791)
    call = _Call(q, lat, g, psi, "half")
    call.run()
    captured = _capture(q, call.run)
    host = torch.from_numpy(U.copy()).pin_memory()
    upload = _capture(q, lambda: g.upload(host))
    b, x = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
    b.upload(psi)
    for k in range(2):
        V = syn.gauge_field(DIMS, 0.3, 1792 + k)
        host.copy_(torch.from_numpy(V))
        _replay(upload)
        call.run()
        assert call.error(V) < 1e-15
        _replay(captured)
        assert call.error(V) < 1e-15
        q.solve_cg(g, x, b, KAPPA, MU, tol=1e-11)
        assert F.rel_err(oracle.apply_m(V, x.download(), KAPPA, MU), psi) < 1e-9


@pytest.mark.parametrize("scale", [1.0, 4.0])
@pytest.mark.parametrize("tps", [0, 1, 8])
def test_first_call_after_an_upload_does_not_wait(q, tps, scale):
    """Operators queued behind an upload that the GPU has not reached return
    at once, and apply the uploaded links, in either form and launch shape (0:
    the library's choice, which is not made by timing such launches)."""
    import time
    import torch
    q.set_hop_threads(tps)
    lat, U, g, psi = _setup(q, seed=1801)
    calls = [_Call(q, lat, g, psi, kind) for kind in ("half", "full", "mhat", "m")]
    ins, outs = ([q.Spinor(lat, p, "f64") for _ in range(3)] for p in ("odd", "even"))
    for s in ins:
        s.upload(syn.to_half(psi, 1))

    def multi():
        q.apply_dslash_multi(g, outs, ins)

    for run in [c.run for c in calls] + [multi]:
        run()
    V = scale * syn.gauge_field(DIMS, 0.3, 1802)
    host = torch.from_numpy(V).pin_memory()
    q.stream_sync()
    torch.cuda._sleep(1_000_000_000)  # half a second at 2 GHz
    t0 = time.perf_counter()
    g.upload(host)
    for run in [c.run for c in calls] + [multi]:
        run()
    waited = time.perf_counter() - t0
    q.stream_sync()
    q.set_hop_threads(0)
    assert waited < 0.5 * (time.perf_counter() - t0)
    for c in calls:
        assert c.error(V) < 1e-15
    for o in outs:
        assert F.rel_err(o.download(), oracle.dhop_eo(V, syn.to_half(psi, 1), 0)) < 1e-15


def test_prepare_leaves_nothing_to_allocate(q):
    """After qcd_gauge_prepare the first F64 operator calls allocate no device
    memory: the free memory stays what it is."""
    import torch
    q.set_hop_threads(0)
    dims = (16, 16, 16, 8)  # 6.4 MB of input workspace
    lat = q.Lattice(dims, -1)
    g = q.Gauge(lat, "f64", 18)
    g.prepare("f64", 18)
    i, o = q.Spinor(lat, "full", "f64"), q.Spinor(lat, "full", "f64")
    q.stream_sync()
    before = torch.cuda.mem_get_info()[0]
    q.apply_dslash(g, o, i)
    q.apply_M(g, o, i, KAPPA, MU)
    q.stream_sync()
    assert torch.cuda.mem_get_info()[0] == before
