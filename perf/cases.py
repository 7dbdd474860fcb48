"""Performance cases of the Wilson / staggered operators and the CG solvers.

Each case is one call that a lattice program makes again and again: a hopping
term or a fermion matrix on resident fields, or a solve.  Lattices follow the
finite-temperature shapes of the workloads (spatial extent about three times
the time extent), from 8^3 x 4 to 48^3 x 12, and ragged ones.

``exact`` computes the same results in complex128 with plain torch: neighbour
tables, gathers and 3x3 matrix products.
"""

import math

import numpy as np
import torch

from paper_1411_5219_gb300 import qcd

# bytes of one site's spinor, and of one real number of a link
_SPINOR_BYTES = {"f64": 192, "f32": 96, "f16": 52, "bf16": 48, "df64": 192}
_KS_BYTES = {"f64": 48, "f32": 24, "f16": 16, "bf16": 12}
_REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "df64": 8}
_PLANES = {"f64": (12, 2, torch.float64), "f32": (6, 4, torch.float32), "f16": (3, 8, torch.float16),
           "bf16": (3, 8, torch.bfloat16), "df64": (12, 4, torch.float32)}
_HOP_FLOPS, _KS_FLOPS = 1320, 570
_KS_PASSES = 8
# even-odd CG iterations to a relative residual of 1e-10 on links exp(0.2 i H)
# at kappa 0.15 to 0.16, for the work of a solve
_ITERATIONS = 40


def listed():
    return [
        # the smallest call: one hopping term of the smallest lattice of a parameter scan, all latency
        dict(name="dslash f64 8x8x8x4", kind="dslash", dims="8x8x8x4", prec="f64", recon=18, dagger=False, full=False),
        # the operator of the double-precision CG at the size of the paper's HMC runs
        dict(name="dslash f64 24x24x24x8", kind="dslash", dims="24x24x24x8", prec="f64", recon=18, dagger=False,
             full=False),
        # the adjoint operator on the largest lattice, in the storage of the mixed-precision inner iterations
        dict(name="dslash f16 48x48x48x12", kind="dslash", dims="48x48x48x12", prec="f16", recon=12, dagger=True,
             full=False),
        # a single-precision measurement on both parities
        dict(name="dslash f32 32x32x32x8", kind="dslash", dims="32x32x32x8", prec="f32", recon=12, dagger=False,
             full=True),
        # the full twisted-mass matrix on a lattice of unequal, ragged extents, as an outer Krylov method calls it
        dict(name="matrix f64 22x18x14x10", kind="matrix", dims="22x18x14x10", prec="f64", recon=18, kappa=0.157,
             mu=0.012, eo=False, dagger=True),
        # the Schur complement on the largest lattice: the true residual of a solve
        dict(name="matrix f64 48x48x48x12", kind="matrix", dims="48x48x48x12", prec="f64", recon=18, kappa=0.16,
             mu=0.01, eo=True, dagger=False),
        # one propagator's spin-colour columns through the operator at once
        dict(name="dslash x12 f32 24x24x24x8", kind="multi", dims="24x24x24x8", prec="f32", recon=12, dagger=False,
             nrhs=12),
        # a polynomial in the staggered operator (here a power of D^2), fetched by the host
        dict(name="staggered f32 32x32x32x8", kind="staggered", dims="32x32x32x8", prec="f32", recon=12),
        # a double-precision solve, the source sent from the host and the solution fetched
        dict(name="solve f64 24x24x24x8", kind="solve", dims="24x24x24x8", inner="f64", recon=18, kappa=0.155, mu=0.0,
             nrhs=1, host=True),
        # the mixed-precision twisted-mass solve of the largest lattice
        dict(name="solve f16 48x48x48x12", kind="solve", dims="48x48x48x12", inner="f16", recon=12, kappa=0.16, mu=0.01,
             nrhs=1, host=False),
        # a propagator and four noise sources as one batch
        dict(name="solve x16 f32 32x32x32x8", kind="solve", dims="32x32x32x8", inner="f32", recon=12, kappa=0.16,
             mu=0.0, nrhs=16, host=False),
        # a scan over couplings on small lattices in one call
        dict(name="scan x12 small", kind="scan", dims="8x8x8x4,12x12x12x4,10x6x8x6,12x12x12x6,8x8x8x8,6x6x6x4", nrhs=12,
             kappa=0.14, mu=0.01),
    ]


def _extents(rng, lo, hi):
    """Even extents of about lo .. hi sites, spread over the logarithm, time the shortest as a rule."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        aspect = rng.uniform(1.0, 4.0)
        nt = (v / aspect ** 3) ** 0.25
        ns = aspect * nt
        d = [max(2, 2 * round(ns * rng.uniform(0.8, 1.25) / 2)) for _ in range(3)] + [max(2, 2 * round(nt / 2))]
        if lo <= d[0] * d[1] * d[2] * d[3] <= hi:
            return "x".join(str(e) for e in d)


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "dslash", "matrix", "matrix", "multi", "staggered", "solve", "solve", "solve",
                       "scan"])
    small, large = 8 * 8 * 8 * 4, 48 * 48 * 48 * 12
    kappa, mu = round(rng.uniform(0.14, 0.16), 4), rng.choice([0.0, round(rng.uniform(0.005, 0.02), 4)])
    if kind == "dslash":
        prec = rng.choice(["f64", "f64", "f32", "f16", "bf16", "df64"])
        recon = 18 if prec in ("f64", "df64") else rng.choice([12, 12, 12, 18])
        return dict(kind=kind, dims=_extents(rng, small, large), prec=prec, recon=recon, dagger=rng.random() < 0.5,
                    full=rng.random() < 0.3)
    if kind == "matrix":
        return dict(kind=kind, dims=_extents(rng, small, large), prec=rng.choice(["f64", "f64", "f32"]), recon=18,
                    kappa=kappa, mu=mu, eo=rng.random() < 0.5, dagger=rng.random() < 0.5)
    if kind == "multi":
        prec = rng.choice(["f64", "f32", "f16"])
        return dict(kind=kind, dims=_extents(rng, small, 24 * 24 * 24 * 8), prec=prec, recon=18 if prec == "f64" else 12,
                    dagger=rng.random() < 0.5, nrhs=rng.randint(2, 16))
    if kind == "staggered":
        prec = rng.choice(["f64", "f32", "f16", "bf16"])
        return dict(kind=kind, dims=_extents(rng, small, 32 * 32 * 32 * 8), prec=prec, recon=18 if prec == "f64" else 12)
    if kind == "solve":
        inner = rng.choice(["f64", "f32", "f16", "f16", "bf16"])
        nrhs = rng.choice([1, 1, 1, rng.randint(2, 12)])
        most = 24 * 24 * 24 * 8 if nrhs > 1 else 32 * 32 * 32 * 8 if inner == "f64" else large
        return dict(kind=kind, dims=_extents(rng, small, most), inner=inner, recon=18 if inner == "f64" else 12,
                    kappa=kappa, mu=mu, nrhs=nrhs, host=nrhs == 1 and rng.random() < 0.4)
    dims = ",".join(_extents(rng, 6 * 6 * 6 * 4, 12 * 12 * 12 * 6) for _ in range(rng.randint(2, 6)))
    return dict(kind="scan", dims=dims, nrhs=rng.randint(6, 16), kappa=round(rng.uniform(0.13, 0.15), 4), mu=mu)


# ------------------------------------------------------------------ inputs


def _dims(text):
    return tuple(int(e) for e in text.split("x"))


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _complex_normal(shape, gen):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=gen))


def _links(dims, seed, stream=1, eps=0.2):
    """SU(3) links exp(i eps H), H Hermitian and traceless with Gaussian entries: [t, z, y, x, mu, 3, 3]."""
    lx, ly, lz, lt = dims
    n = 4 * lx * ly * lz * lt
    gen = _generator(seed, stream)
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    for s in range(0, n, 1 << 20):
        m = min(1 << 20, n - s)
        a = _complex_normal((m, 3, 3), gen)
        h = 0.5 * (a + a.mH)
        h = h - (h.diagonal(dim1=1, dim2=2).sum(-1) / 3)[:, None, None] * torch.eye(3, dtype=h.dtype, device="cuda")
        out[s:s + m] = torch.linalg.matrix_exp(1j * eps * h)
    return out.view(lt, lz, ly, lx, 4, 3, 3)


def _source(dims, seed, k, inner=(4, 3)):
    lx, ly, lz, lt = dims
    return _complex_normal((lt, lz, ly, lx) + inner, _generator(seed, 100 + k))


def _point(dims, k):
    """Source k of a propagator: 1 in spin-colour component k at a site off the corner."""
    lx, ly, lz, lt = dims
    b = torch.zeros(lt, lz, ly, lx, 12, dtype=torch.complex128, device="cuda")
    b[lt // 2, lz // 2, 1, lx // 2, k] = 1.0
    return b.view(lt, lz, ly, lx, 4, 3)


def _sources(case, dims, seed):
    """The sources of a solve: a batch of more than twelve starts with a propagator's columns."""
    n = case["nrhs"]
    return [_point(dims, k) if n > 12 and k < 12 else _source(dims, seed, k) for k in range(n)]


def _scan(case):
    """The systems of a scan: extents, hopping parameter and twisted mass of each."""
    lattices = [_dims(t) for t in case["dims"].split(",")]
    n = case["nrhs"]
    return [(lattices[k % len(lattices)], case["kappa"] + 0.015 * k / n, case["mu"] if k % 2 else 0.0) for k in range(n)]


def _parity(dims):
    lx, ly, lz, lt = dims
    t, z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in (lt, lz, ly, lx)], indexing="ij")
    return ((x + y + z + t) % 2).reshape(-1)


def _half(full, dims, p):
    return full.reshape(-1, *full.shape[4:])[_parity(dims) == p].contiguous()


def _planes(spinor, lat, prec, full):
    """The device planes of a spinor over torch memory, without the padding: [half, plane, site, reals] (and FP16 scales)."""
    n, width, dtype = _PLANES[prec]
    h = lat.volume // 2
    data, norm = spinor._buffers
    nh = 2 if full else 1
    planes = data.view(dtype).view(nh, n, -1, width)[:, :, :h]
    return {"data": planes, "scale": norm.view(torch.float32).view(nh, -1)[:, :h]} if prec == "f16" else {"data": planes}


def prepare(case, seed):
    if case["kind"] == "scan":
        systems = []
        for k, (dims, kappa, mu) in enumerate(_scan(case)):
            lat = qcd.Lattice(dims, -1)
            g = qcd.Gauge(lat, "f64", 18)
            g.upload(_links(dims, seed, 10 + k).cpu())
            b, x = qcd.Spinor(lat, "full", "f64"), qcd.Spinor(lat, "full", "f64", torch_alloc=True)
            b.upload(_source(dims, seed, k).cpu())
            qcd.stream_sync()
            systems.append((g, x, b, kappa, mu, _planes(x, lat, "f64", True)))
        return {"case": case, "g": [s[0] for s in systems], "x": [s[1] for s in systems], "b": [s[2] for s in systems],
                "kappa": [s[3] for s in systems], "mu": [s[4] for s in systems], "out": [s[5] for s in systems]}
    dims = _dims(case["dims"])
    lat = qcd.Lattice(dims, -1)
    g = qcd.Gauge(lat, "f64", case["recon"])
    g.upload(_links(dims, seed).cpu())
    s = {"case": case, "lat": lat, "g": g}
    if case["kind"] == "solve":
        if case["inner"] != "f64":
            g.prepare(case["inner"], case["recon"])
        s["x"] = [qcd.Spinor(lat, "full", "f64", torch_alloc=True) for _ in range(case["nrhs"])]
        s["b"] = [qcd.Spinor(lat, "full", "f64") for _ in range(case["nrhs"])]
        host = [b.cpu().pin_memory() if case["host"] else b.cpu() for b in _sources(case, dims, seed)]
        for field, b in zip(s["b"], host):
            field.upload(b)
        qcd.stream_sync()
        if case["host"]:
            s["b_host"], s["x_host"] = host[0], torch.empty_like(host[0]).pin_memory()
        s["out"] = [_planes(x, lat, "f64", True) for x in s["x"]]
        return s
    prec = case["prec"]
    g.prepare(prec, case["recon"])
    if case["kind"] == "staggered":
        s["even"], s["odd"] = (qcd.Spinor(lat, p, prec, ks=True) for p in ("even", "odd"))
        s["chi"] = qcd.Spinor(lat, "even", prec, ks=True)
        s["chi"].upload(_half(_source(dims, seed, 0, (3,)), dims, 0).cpu())
        s["host"] = torch.empty(s["chi"].host_shape, dtype=torch.complex128).pin_memory()
        qcd.stream_sync()
        return s
    full = case["full"] if case["kind"] == "dslash" else not case["eo"] if case["kind"] == "matrix" else False
    parity_in = "full" if full else "even" if case["kind"] == "matrix" else "odd"
    parity_out = "full" if full else "even"
    n = case.get("nrhs", 1)
    s["in"] = [qcd.Spinor(lat, parity_in, prec) for _ in range(n)]
    s["out_fields"] = [qcd.Spinor(lat, parity_out, prec, torch_alloc=True) for _ in range(n)]
    for k, field in enumerate(s["in"]):
        psi = _source(dims, seed, k)
        field.upload((psi if full else _half(psi, dims, 0 if parity_in == "even" else 1)).cpu())
    qcd.stream_sync()
    if prec == "df64":  # a program goes on in double precision
        s["f64"] = qcd.Spinor(lat, parity_out, "f64", torch_alloc=True)
        s["out"] = [_planes(s["f64"], lat, "f64", full)]
    else:
        s["out"] = [_planes(f, lat, prec, full) for f in s["out_fields"]]
    return s


# ------------------------------------------------------------------ the calls


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "dslash":
        qcd.apply_dslash(s["g"], s["out_fields"][0], s["in"][0], dagger=c["dagger"])
        if c["prec"] == "df64":
            s["f64"].convert_from(s["out_fields"][0])
    elif kind == "matrix":
        qcd.apply_M(s["g"], s["out_fields"][0], s["in"][0], c["kappa"], c["mu"], eo=c["eo"], dagger=c["dagger"])
    elif kind == "multi":
        qcd.apply_dslash_multi(s["g"], s["out_fields"], s["in"], dagger=c["dagger"])
    elif kind == "staggered":
        src = s["chi"]
        for _ in range(_KS_PASSES):
            qcd.apply_dslash_ks(s["g"], s["odd"], src)
            qcd.apply_dslash_ks(s["g"], s["even"], s["odd"])
            src = s["even"]
        return s["even"].download(s["host"])
    elif kind == "scan":
        qcd.solve_cg_many(s["g"], s["x"], s["b"], s["kappa"], s["mu"])
    elif c["nrhs"] > 1:
        qcd.solve_cg_multi(s["g"], s["x"], s["b"], c["kappa"], c["mu"], inner_prec=c["inner"], inner_recon=c["recon"])
    else:
        if c["host"]:
            s["b"][0].upload(s["b_host"])
        qcd.solve_cg(s["g"], s["x"][0], s["b"][0], c["kappa"], c["mu"], inner_prec=c["inner"], inner_recon=c["recon"])
        if c["host"]:
            return s["x"][0].download(s["x_host"])
    return s["out"]


def work(case):
    kind = case["kind"]
    if kind == "scan":
        total = sum(d[0] * d[1] * d[2] * d[3] for d, _, _ in _scan(case))
        sites = 4 * _ITERATIONS * total / 2
        return {"bytes": sites * (8 * 144 + 2 * 192), "flops": sites * _HOP_FLOPS}
    d = _dims(case["dims"])
    h = d[0] * d[1] * d[2] * d[3] / 2
    n = case.get("nrhs", 1)
    if kind == "solve":
        p = case["inner"]
        hops = 4 * _ITERATIONS
        link = 8 * case["recon"] * _REAL_BYTES[p]
        return {"bytes": hops * h * (link + 2 * n * _SPINOR_BYTES[p]), "flops": hops * h * n * _HOP_FLOPS}
    link = 8 * case["recon"] * _REAL_BYTES[case["prec"]]
    if kind == "staggered":
        hops = 2 * _KS_PASSES
        return {"bytes": hops * h * (link + 2 * _KS_BYTES[case["prec"]]), "flops": hops * h * _KS_FLOPS}
    site = _SPINOR_BYTES[case["prec"]]
    if kind == "matrix":  # both parities, or two hops of which the second reads the input again
        return {"bytes": 2 * h * (link + 2 * site) + (h * site if case["eo"] else 0), "flops": 2 * h * _HOP_FLOPS}
    halves = 2 if case.get("full") else 1
    return {"bytes": halves * h * (link + 2 * n * site), "flops": halves * h * n * _HOP_FLOPS}


def tolerance(case):
    if case["kind"] == "scan":
        return {"rel": 2e-9}  # the solution at a relative residual of 1e-10
    if case["kind"] == "solve":
        return {"rel": 2e-9}
    # one rounding of each input, link and result in the storage format (and
    # the rounding of the sums, of the same size in 32 and 64 bits); the
    # staggered power takes sixteen of them
    prec = case["prec"]
    u = {"f64": 2.0 ** -53, "df64": 2.0 ** -48, "f32": 2.0 ** -24, "f16": 2.0 ** -11, "bf16": 2.0 ** -8}[prec]
    return {"rel": min(0.03, (16 if case["kind"] == "staggered" else 4 if prec in ("f16", "bf16") else 8) * u)}


# ------------------------------------------------------------------ the same in 64 bits

_SIGMA = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]


def _gamma():
    """Chiral basis: gamma_k = [[0, -i sigma_k], [i sigma_k, 0]], gamma_4 = [[0, 1], [1, 0]]."""
    z = np.zeros((2, 2))
    g = [np.block([[z, -1j * np.array(s)], [1j * np.array(s), z]]) for s in _SIGMA]
    return g + [np.block([[z, np.eye(2)], [np.eye(2), z]])]


class _Operator:
    """Hopping terms between half fields [site / 2, ...]: neighbour tables and the link of each of the eight hops."""

    def __init__(self, u, dims, staggered=False):
        lx, ly, lz, lt = dims
        v = lx * ly * lz * lt
        u = u.reshape(v, 4, 3, 3)
        lex = torch.arange(v, device="cuda")
        x, y, z, t = lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)
        self.par = (x + y + z + t) % 2
        self.sites = [lex[self.par == p] for p in (0, 1)]
        self.spin = [[torch.from_numpy(np.eye(4) + sign * g).to("cuda", torch.complex128) for sign in (-1, 1)]
                     for g in _gamma()]
        one = torch.ones_like(lex)
        eta = [one, 1 - 2 * (x % 2), 1 - 2 * ((x + y) % 2), 1 - 2 * ((x + y + z) % 2)]
        step, size, at = (1, lx, lx * ly, lx * ly * lz), dims, (x, y, z, t)
        self.hops = ([], [])
        for p in (0, 1):
            s = self.sites[p]
            for mu in range(4):
                a, n = at[mu][s], size[mu]
                for back in (0, 1):
                    wrap = a == 0 if back else a == n - 1
                    nb = s + (torch.where(wrap, n - 1, -1) if back else torch.where(wrap, 1 - n, 1)) * step[mu]
                    m = u[nb, mu].mH if back else u[s, mu]
                    sign = torch.where(wrap, -1.0, 1.0) if mu == 3 else torch.ones(len(s), device="cuda")
                    if staggered:
                        sign = sign * eta[mu][s] * (1 - 2 * back)
                    self.hops[p].append((mu, back, nb // 2, m * sign[:, None, None]))

    def hop(self, p, other, dagger=False):
        """The sites of parity p from the half field of the other parity."""
        out = None
        for mu, back, nb, m in self.hops[p]:
            v = torch.einsum("st,ntc->nsc", self.spin[mu][back != dagger], other[nb]) if other.dim() == 3 else other[nb][:, None]
            v = torch.matmul(v, m.mT)
            out = v if out is None else out.add_(v)
        return out if other.dim() == 3 else out[:, 0]

    def halves(self, full):
        f = full.reshape(-1, *full.shape[4:])
        return [f[s] for s in self.sites]

    @staticmethod
    def twist(v, a, inverse=False):
        f = torch.tensor([1 + 1j * a, 1 + 1j * a, 1 - 1j * a, 1 - 1j * a], device="cuda", dtype=torch.complex128)
        return v * (1 / f if inverse else f)[None, :, None]

    def schur(self, v, kappa, a, dagger=False):
        b = -a if dagger else a
        t = self.twist(self.hop(1, v, dagger), b, True)
        return self.twist(v, b) - kappa ** 2 * self.hop(0, t, dagger)

    def solve(self, b, kappa, mu):
        """[even, odd] of x with M x = b, by even-odd CG on the normal equations to rounding."""
        a = 2 * kappa * mu
        be, bo = self.halves(b)
        rhs = self.schur(be + kappa * self.hop(0, self.twist(bo, a, True)), kappa, a, True)
        x, r = torch.zeros_like(rhs), rhs.clone()
        p, rr = r.clone(), float(torch.linalg.vector_norm(r)) ** 2
        stop = 1e-28 * rr
        for _ in range(300):
            if rr <= stop:
                break
            m = self.schur(p, kappa, a)
            alpha = rr / float(torch.linalg.vector_norm(m)) ** 2
            x += alpha * p
            r -= alpha * self.schur(m, kappa, a, True)
            new = float(torch.linalg.vector_norm(r)) ** 2
            p = r + (new / rr) * p
            rr = new
        return [x, self.twist(bo + kappa * self.hop(1, x), a, True)]


def _laid_out(halves, prec):
    """Half fields [site, 4, 3] as device planes, in 64 bits."""
    n, width, _ = _PLANES[prec]
    v = torch.stack([torch.view_as_real(h.resolve_conj().contiguous()).reshape(len(h), 24) for h in halves])
    out = {}
    if prec == "f16":
        out["scale"] = v.abs().amax(-1)
        v = v / out["scale"][..., None]
    out["data"] = v.view(v.shape[0], v.shape[1], n, width).transpose(1, 2)
    return out


def _lexicographic(halves, op, dims):
    lx, ly, lz, lt = dims
    full = torch.empty(lx * ly * lz * lt, 4, 3, dtype=torch.complex128, device="cuda")
    for s, h in zip(op.sites, halves):
        full[s] = h
    return full.view(lt, lz, ly, lx, 4, 3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        out = []
        for k, (dims, kappa, mu) in enumerate(_scan(case)):
            op = _Operator(_links(dims, seed, 10 + k), dims)
            out.append(_laid_out(op.solve(_source(dims, seed, k), kappa, mu), "f64"))
        return out
    dims = _dims(case["dims"])
    op = _Operator(_links(dims, seed), dims, kind == "staggered")
    if kind == "solve":
        if case["host"]:
            return _lexicographic(op.solve(_source(dims, seed, 0), case["kappa"], case["mu"]), op, dims)
        return [_laid_out(op.solve(b, case["kappa"], case["mu"]), "f64") for b in _sources(case, dims, seed)]
    if kind == "staggered":
        v = _half(_source(dims, seed, 0, (3,)), dims, 0)
        for _ in range(_KS_PASSES):
            v = op.hop(0, op.hop(1, v))
        return v
    prec = "f64" if case["prec"] == "df64" else case["prec"]
    out = []
    for k in range(case.get("nrhs", 1)):
        e, o = op.halves(_source(dims, seed, k))
        if kind == "matrix":
            a = 2 * case["kappa"] * case["mu"]
            if case["eo"]:
                halves = [op.schur(e, case["kappa"], a, case["dagger"])]
            else:
                b = -a if case["dagger"] else a
                halves = [op.twist(v, b) - case["kappa"] * op.hop(p, w, case["dagger"])
                          for p, v, w in ((0, e, o), (1, o, e))]
        elif case.get("full"):
            halves = [op.hop(0, o, case["dagger"]), op.hop(1, e, case["dagger"])]
        else:
            halves = [op.hop(0, o, case["dagger"])]
        out.append(_laid_out(halves, prec))
    return out
