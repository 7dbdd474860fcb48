"""qcd_apply_dslash_multi on fields where they lie: full lattices, group
remainders, and outputs that are another right-hand side's input (gathered
first, as one batch), against the FP64 oracle at the storage tolerances."""

import numpy as np
import pytest

import oracle
from paper_1411_5219_gb300 import synthetic as syn
from tests import _fields as F

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-15, "f32": 8 * 2.0 ** -24, "f16": 8 * 2.0 ** -11, "bf16": 8 * 2.0 ** -8}


@pytest.fixture(scope="module")
def q():
    from paper_1411_5219_gb300 import _build, qcd
    _build.build()
    import torch
    assert torch.cuda.is_available()
    return qcd


@pytest.mark.parametrize("prec,recon", [("f64", 18), ("f64", 12), ("f32", 12), ("f32", 18), ("f16", 12), ("bf16", 8)])
@pytest.mark.parametrize("nrhs", [1, 3, 6, 11, 32])
def test_multi_full_lattice(q, prec, recon, nrhs):
    dims = (6, 2, 4, 10)  # 240 sites a parity: a ragged last block
    lat = q.Lattice(dims, -1)
    U = syn.gauge_field(dims, 0.2, 1601)
    g = q.Gauge(lat, "f64", recon)
    g.upload(U)
    psi = [syn.gaussian_spinor(dims, 1610 + k) for k in range(nrhs)]
    ins, outs = ([q.Spinor(lat, "full", prec) for _ in psi] for _ in range(2))
    for s, v in zip(ins, psi):
        s.upload(v)
    q.apply_dslash_multi(g, outs, ins, dagger=True)
    for k, v in enumerate(psi):
        assert F.rel_err(outs[k].download(), oracle.dhop(U, v, dagger=True)) <= TOL[prec], k


@pytest.mark.parametrize("prec,recon", [("f64", 18), ("f32", 12)])
def test_multi_output_is_another_input(q, prec, recon):
    dims = (4, 4, 2, 4)
    lat = q.Lattice(dims, -1)
    U = syn.gauge_field(dims, 0.2, 1602)
    g = q.Gauge(lat, "f64", recon)
    g.upload(U)
    psi = [syn.gaussian_spinor(dims, 1630 + k) for k in range(3)]
    ins = [q.Spinor(lat, "full", prec) for _ in psi]
    for s, v in zip(ins, psi):
        s.upload(v)
    q.apply_dslash_multi(g, ins[1:] + ins[:1], ins)
    for k, v in enumerate(psi):
        assert F.rel_err(ins[(k + 1) % 3].download(), oracle.dhop(U, v)) <= TOL[prec], k


@pytest.mark.parametrize("staggered", ["in", "out"])
def test_multi_rejects_staggered_fields(q, staggered):
    """Three complex a site instead of twelve: refused, not read past their end."""
    lat = q.Lattice((4, 4, 2, 4), -1)
    g = q.Gauge(lat, "f64", 18)
    ins = [q.Spinor(lat, "odd", "f32", ks=staggered == "in" and k == 1) for k in range(2)]
    outs = [q.Spinor(lat, "even", "f32", ks=staggered == "out" and k == 1) for k in range(2)]
    with pytest.raises(q.QcdError) as e:
        q.apply_dslash_multi(g, outs, ins)
    assert e.value.status == 1
