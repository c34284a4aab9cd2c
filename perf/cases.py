"""The work that users of this library have it do, as cases that can be timed.

Each case is one call sequence of the Python binding, the way a program makes it:
links sit in a gauge field that the program keeps (with the plans that the library
keeps for it), sources arrive as CUDA complex128 tensors in the canonical order,
results leave the same way or stay in the caller's field.  Sizes are those of the
workloads, tests and benchmark of this repository, or generic ones.
"""
from __future__ import annotations

import math

import torch

from paper_2001_05218_gb300 import autograd, dw, inputs

# hopping parameter and link ensemble of the 16^3 x 32 workload
USUAL = dict(kappa=0.124, links="exp", amplitude=0.4)


def listed():
    c = USUAL
    return [
        # one small system with the default parameters (FP32 inner, IEEE-FP64 outer): latency
        dict(c, name="solve_4x4x4x4_defaults", what="solve", lx=4, ly=4, lz=4, lt=4, links="haar", kappa=0.12,
             inner="f32", outer="f64", compress12=0, nrhs=1),
        # the ordinary lattice of the workloads, the benchmark's precisions
        dict(c, name="solve_16x16x16x32_f16", what="solve", lx=16, ly=16, lz=16, lt=32, inner="f16", outer="df64",
             compress12=1, nrhs=1),
        # extents that are no powers of two and differ in every direction, FP32 inner
        dict(c, name="solve_20x12x18x30_f32", what="solve", lx=20, ly=12, lz=18, lt=30, inner="f32", outer="df64",
             compress12=0, nrhs=1),
        # the headline workload: time to 1e-10 on the largest lattice
        dict(c, name="solve_32x32x32x64_f16", what="solve", lx=32, ly=32, lz=32, lt=64, amplitude=0.6, kappa=0.1245,
             inner="f16", outer="df64", compress12=1, nrhs=1),
        # a quark propagator: the 12 spin-colour point sources of one site
        dict(c, name="propagator_24x24x24x48", what="solve", lx=24, ly=24, lz=24, lt=48, kappa=0.119, inner="f16",
             outer="df64", compress12=1, nrhs=12),
        # independent lattices of different sizes solved together
        dict(c, name="batch_of_8_lattices", what="batch", count=8, scale=1.0, inner="f16", outer="df64", compress12=1),
        # pseudofermion action and its gradients (forward, adjoint, force), as in molecular dynamics
        dict(c, name="action_gradient_16x16x16x32", what="gradient", lx=16, ly=16, lz=16, lt=32, kappa=0.12,
             inner="f32", outer="df64", compress12=0),
        # the second stencil's solver
        dict(c, name="laplace_solve_16x16x16x32", what="laplace", lx=16, ly=16, lz=16, lt=32, inner="f32",
             outer="df64", compress12=0),
        # single operator applications, as a caller's own solver makes them: the smallest ...
        dict(c, name="apply_8x8x8x8_f32_even", what="apply", lx=8, ly=8, lz=8, lt=8, prec="f32", compress12=0,
             kind="even", op="apply", nrhs=1),
        # ... the reference precision, both parities, D^dag D ...
        dict(c, name="normal_16x16x16x32_f64_full", what="apply", lx=16, ly=16, lz=16, lt=32, prec="f64",
             compress12=0, kind="full", op="normal", nrhs=1),
        # ... the double-float operator (high-precision residuals) at a middle size ...
        dict(c, name="dag_24x24x24x48_df64_even", what="apply", lx=24, ly=24, lz=24, lt=48, prec="df64",
             compress12=0, kind="even", op="dag", nrhs=1),
        # ... and the 16-bit operator on the largest lattice
        dict(c, name="apply_32x32x32x64_f16_even", what="apply", lx=32, ly=32, lz=32, lt=64, amplitude=0.6,
             kappa=0.1245, prec="f16", compress12=1, kind="even", op="apply", nrhs=1),
    ]


def draw(rng):
    """One more case of the same ranges."""
    what = rng.choice(["solve", "solve", "solve", "solve", "batch", "gradient", "laplace", "apply", "apply", "apply",
                       "apply"])
    c = dict(what=what, links="exp", kappa=round(rng.uniform(0.115, 0.124), 5),
             amplitude=round(rng.uniform(0.4, 0.6), 3))
    if rng.random() < 0.1:
        c.update(links="haar", kappa=round(rng.uniform(0.115, 0.12), 5))
    if what == "batch":
        c.update(count=rng.randint(2, 8), scale=rng.choice([0.5, 0.75, 1.0]), outer="df64")
        c.update(rng.choice([dict(inner="f16", compress12=1), dict(inner="f32", compress12=0)]))
        return c
    nrhs = 1
    if what in ("solve", "apply") and rng.random() < 0.3:
        nrhs = rng.choice([2, 3, 4, 6, 8, 12])
    top = {"solve": 1.8e6, "apply": 1.8e6, "gradient": 1.4e5, "laplace": 1.0e6}[what] / nrhs
    volume = math.exp(rng.uniform(math.log(256.0), math.log(top)))
    dims = [4, 4, 4, 4]
    while dims[0] * dims[1] * dims[2] * dims[3] < volume:
        dims[rng.randrange(4)] += 2
    while (dims[0] * dims[1] * dims[2] * dims[3]) % 16:
        dims[rng.randrange(4)] += 2
    if rng.random() < 0.5:  # time is often the longest direction
        dims.sort()
    c.update(lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3])
    if what == "solve":
        c.update(rng.choice([dict(inner="f16", compress12=1), dict(inner="f16", compress12=1),
                             dict(inner="f32", compress12=0), dict(inner="f32", compress12=1),
                             dict(inner="bf16", compress12=1), dict(inner="i16", compress12=1)]))
        c.update(outer=rng.choice(["df64", "df64", "f64"]), nrhs=nrhs)
        if c["outer"] == "f64" and volume * nrhs > 2e5:
            c["outer"] = "df64"
    elif what == "apply":
        c.update(rng.choice([dict(prec="f64", compress12=0), dict(prec="f32", compress12=0),
                             dict(prec="f32", compress12=1), dict(prec="f16", compress12=1),
                             dict(prec="f16", compress12=0), dict(prec="bf16", compress12=1),
                             dict(prec="df64", compress12=0)]))
        c.update(kind=rng.choice(["even", "odd", "full"]), op=rng.choice(["apply", "dag", "normal", "norm"]),
                 nrhs=nrhs)
    else:
        c.update(inner="f32", outer="df64", compress12=0)
    return c


# ------------------------------------------------------------------ inputs
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 62))


def _gaussian(g, *shape):
    return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=g) * math.sqrt(2.0)


def _mul3(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _exp_links(g, n, amplitude):
    """exp(i a H), H random traceless Hermitian."""
    a = torch.randn(n, 3, 3, dtype=torch.complex128, device="cuda", generator=g)
    h = 0.5 * (a + a.mH)
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    h = h - (h.diagonal(dim1=1, dim2=2).sum(-1).real / 3.0)[:, None, None] * eye
    x = h * (1j * amplitude / 16.0)
    u = eye + x
    term = x
    for k in range(2, 13):
        term = _mul3(term, x) / k
        u = u + term
    for _ in range(4):
        u = _mul3(u, u)
    return u


def _haar_links(g, n):
    a = torch.randn(n, 3, 3, dtype=torch.complex128, device="cuda", generator=g)
    rows = []
    for i in range(3):
        v = a[:, i]
        for _ in range(2):
            for w in rows:
                v = v - (w.conj() * v).sum(-1, keepdim=True) * w
        rows.append(v / v.abs().square().sum(-1, keepdim=True).sqrt())
    u = torch.stack(rows, 1)
    det = (u[:, 0] * torch.linalg.cross(u[:, 1], u[:, 2])).sum(-1)
    ang = torch.angle(det) / -3.0
    return u * torch.polar(torch.ones_like(ang), ang)[:, None, None]


def _links(c, dims, seed):
    g = _generator(seed)
    n = 4 * inputs.volume(dims)
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    for i in range(0, n, 1 << 20):
        m = min(1 << 20, n - i)
        out[i:i + m] = _haar_links(g, m) if c["links"] == "haar" else _exp_links(g, m, c["amplitude"])
    return out.view(-1, 4, 3, 3)


def _source(dims, seed, nrhs):
    """A Gaussian source, or with several right-hand sides the spin-colour point sources of one site."""
    V = inputs.volume(dims)
    g = _generator(seed + (1 << 40))
    if nrhs == 1:
        return _gaussian(g, V, 4, 3)
    b = torch.zeros(nrhs, V, 4, 3, dtype=torch.complex128, device="cuda")
    site = int(torch.randint(V, (1,), generator=g, device="cuda"))
    for r in range(nrhs):
        b[r, site, (r // 3) % 4, r % 3] = 1.0
    return b


def _gauge(c, dims, seed, kappa, prec=dw.DW_F64, compress12=0):
    f = dw.Field(dw.lattice(dims, kappa), dw.DW_GAUGE, prec, compress12)
    U = _links(c, dims, seed)
    f.import_(U)
    return f, U


def _spinor(dims, kind=dw.DW_SPINOR_FULL, prec=dw.DW_F64, nrhs=1):
    return dw.Field(dw.lattice(dims), kind, prec, 0, nrhs)


def _params(c):
    return dw.params(tol=1e-10, inner=c["inner"], outer=c["outer"], compress12=c["compress12"])


KINDS = {"even": dw.DW_SPINOR_EVEN, "odd": dw.DW_SPINOR_ODD, "full": dw.DW_SPINOR_FULL}


def _batch(c, seed):
    for i in range(c["count"]):
        dims = tuple(max(4, 2 * round(c["scale"] * d / 2)) for d in inputs.RAGGED_DIMS[i])
        yield dims, 0.115 + 0.01 * ((i * 5 + 2) % 9) / 9.0, seed * 16 + i


def prepare(case, seed):
    c = case
    what = c["what"]
    if what == "batch":
        s = dict(U=[], b=[], bf=[], xf=[])
        for dims, kappa, k in _batch(c, seed):
            s["U"].append(_gauge(c, dims, k, kappa)[0])
            s["b"].append(_source(dims, k, 1))
            s["bf"].append(_spinor(dims))
            s["xf"].append(_spinor(dims))
        return dict(s, what=what, p=_params(c))
    dims = _dims(c)
    if what == "gradient":
        return dict(what=what, lat=dw.lattice(dims, c["kappa"]), U=_links(c, dims, seed).requires_grad_(),
                    phi=_source(dims, seed, 1).requires_grad_(), p=_params(c))
    if what == "apply":
        prec, kind = dw.PREC[c["prec"]], KINDS[c["kind"]]
        U, _ = _gauge(c, dims, seed, c["kappa"], prec, c["compress12"])
        x, y = (_spinor(dims, kind, prec, c["nrhs"]) for _ in range(2))
        x.import_(_apply_input(c, seed))
        return dict(what=what, U=U, x=x, y=y, op=c["op"])
    U, _ = _gauge(c, dims, seed, c["kappa"])
    nrhs = c.get("nrhs", 1)
    return dict(what=what, U=U, b=_source(dims, seed, nrhs), bf=_spinor(dims, nrhs=nrhs),
                xf=_spinor(dims, nrhs=nrhs), p=_params(c))


def _apply_input(c, seed):
    V, nrhs = inputs.volume(_dims(c)), c["nrhs"]
    n = V if c["kind"] == "full" else V // 2
    return _gaussian(_generator(seed + (1 << 41)), *((nrhs, n, 4, 3) if nrhs > 1 else (n, 4, 3)))


# ------------------------------------------------------------------ one pass
def _own_memory(f):
    """The field's memory as its numbers (double-float fields as complex128)."""
    if f.prec == dw.DW_DF64:
        return f.export()
    raw = f.storage[f.offset:f.offset + f.nbytes]
    if f.prec in (dw.DW_F64, dw.DW_F32):
        return raw.view(torch.float64 if f.prec == dw.DW_F64 else torch.float32)
    block = raw.view(-1, 26 * int(math.prod(list(f.lat.dims))))  # one parity of one right-hand side
    half = block.shape[1] // 13 * 12
    numbers = torch.float16 if f.prec == dw.DW_F16 else torch.bfloat16
    return [block[:, :half].view(numbers), block[:, half:].view(torch.float32)]


def run(state):
    s = state
    what = s["what"]
    if what == "apply":
        if s["op"] == "norm":
            return [dw.apply_norm(s["U"], s["x"], s["y"]), _own_memory(s["y"])]
        dw.apply(s["U"], s["x"], s["y"], dag=s["op"] == "dag", normal=s["op"] == "normal")
        return _own_memory(s["y"])
    if what == "gradient":
        s["U"].grad = s["phi"].grad = None
        S = autograd.PseudofermionAction.apply(s["U"], s["phi"], s["lat"], s["p"])
        S.backward()
        return [S.detach(), s["U"].grad, s["phi"].grad]
    if what == "batch":
        for b, bf, xf in zip(s["b"], s["bf"], s["xf"]):
            bf.import_(b)
            xf.storage.zero_()
        dw.cg_solve_batched(s["U"], s["bf"], s["xf"], s["p"])
        return [xf.export() for xf in s["xf"]]
    s["bf"].import_(s["b"])
    s["xf"].storage.zero_()
    (dw.cg_solve_laplace if what == "laplace" else dw.cg_solve)(s["U"], s["bf"], s["xf"], s["p"])
    return s["xf"].export()


# ------------------------------------------------------------------ work
LINK = {"f64": (144, 96), "df64": (144, 96), "f32": (72, 48), "f16": (36, 24), "bf16": (36, 24)}
SPIN = {"f64": 192, "df64": 192, "f32": 96, "f16": 52, "bf16": 52}


def work(case):
    """Links and source read once and the result written once; a solve's operations are those of an estimated
    60 iterations (20 for the Laplacian) of four parity hops, 1320 each (2280 for the Laplacian)."""
    c = case
    if c["what"] == "batch":
        sites = sum(inputs.volume(d) for d, _, _ in _batch(c, 0))
        return {"bytes": 960.0 * sites, "flops": 60 * 2 * 1320.0 * sites}
    sites = inputs.volume(_dims(c))
    nrhs = c.get("nrhs", 1)
    if c["what"] == "apply":
        part = 1.0 if c["kind"] == "full" else 0.5
        hops = sites * (2 if c["op"] == "normal" else 1)
        return {"bytes": sites * (4.0 * LINK[c["prec"]][c["compress12"]] + 2 * part * nrhs * SPIN[c["prec"]]),
                "flops": 1320.0 * hops * nrhs}
    if c["what"] == "gradient":
        return {"bytes": (2 * 576.0 + 2 * 192) * sites, "flops": 2 * 120 * 2 * 1320.0 * sites}
    if c["what"] == "laplace":
        return {"bytes": 960.0 * sites, "flops": 20 * 2280.0 * sites}
    return {"bytes": (576.0 + 384 * nrhs) * sites, "flops": 60 * 2 * 1320.0 * sites * nrhs}


# ------------------------------------------------------------------ the same in 64 bits
# gamma_mu psi: spin s takes FACTOR[mu][s] * psi[SPIN_OF[mu][s]]
SPIN_OF = [(3, 2, 1, 0), (3, 2, 1, 0), (2, 3, 0, 1), (2, 3, 0, 1)]
FACTOR = [(-1j, -1j, 1j, 1j), (-1, 1, 1, -1), (-1j, 1j, 1j, -1j), (1, 1, 1, 1)]


def _shift(p, mu, step):
    """psi(x + step mu), with the sign of the antiperiodic time direction; p: (n, t, z, y, x, ...)."""
    q = torch.roll(p, -step, dims=4 - mu)
    if mu == 3:
        q[:, -1 if step > 0 else 0] *= -1
    return q


def _times(u, p):
    """u (n, t, z, y, x, a, b) on the colours of p (n, t, z, y, x, spin, colour)."""
    return sum(u[..., None, :, b] * p[..., b, None] for b in range(3))


def _gamma(p, mu):
    f = torch.tensor(FACTOR[mu], dtype=torch.complex128, device=p.device)
    return p[..., list(SPIN_OF[mu]), :] * f[:, None]


def _grid(t, dims, tail):
    return t.reshape(-1, dims[3], dims[2], dims[1], dims[0], *tail)


def _hopping(U, p, sign, laplace=False):
    """sum_mu (1 - sign gamma) U psi(x + mu) + (1 + sign gamma) U^dag(x - mu) psi(x - mu)."""
    out = torch.zeros_like(p)
    for mu in range(4):
        u = U[..., mu, :, :]
        f = _shift(p, mu, 1)
        f = _times(u, f if laplace else f - sign * _gamma(f, mu))
        b = _times(u.mH, p if laplace else p + sign * _gamma(p, mu))
        out += f + _shift(b, mu, -1)
    return out


def _operator(U, kappa, laplace=False):
    return lambda p, sign=1: p - kappa * _hopping(U, p, sign, laplace)


def _cg(A, b, tol=1e-14, most=4000):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r, r.abs().square().sum()
    stop = rr * tol * tol
    for _ in range(most):
        w = A(p)
        a = rr / (p.conj() * w).sum().real
        x = x + a * p
        r = r - a * w
        new = r.abs().square().sum()
        if new <= stop:
            break
        p = r + (new / rr) * p
        rr = new
    return x


def _solution(c, dims, kappa, seed, nrhs, laplace=False):
    U = _grid(_links(c, dims, seed), dims, (4, 3, 3))
    b = _source(dims, seed, nrhs)
    D = _operator(U, kappa, laplace)
    g = _grid(b, dims, (4, 3))
    x = _cg(D, g) if laplace else _cg(lambda p: D(D(p), -1), D(g, -1))
    return x.reshape(b.shape)


def exact(case, seed):
    c = case
    if c["what"] == "batch":
        return [_solution(c, dims, kappa, k, 1) for dims, kappa, k in _batch(c, seed)]
    dims = _dims(c)
    V = inputs.volume(dims)
    if c["what"] == "apply":
        return _exact_apply(c, dims, seed)
    if c["what"] == "gradient":
        U = _grid(_links(c, dims, seed), dims, (4, 3, 3))
        phi = _grid(_source(dims, seed, 1), dims, (4, 3))
        D = _operator(U, c["kappa"])
        X = _cg(lambda p: D(D(p), -1), phi)
        Y = D(X)
        V1 = U.clone().requires_grad_()
        # dS = -2 Re <Y, dD X>
        (-2.0 * (Y.conj() * _operator(V1, c["kappa"])(X)).sum().real).backward()
        return [(phi.conj() * X).sum().real, V1.grad.reshape(V, 4, 3, 3), (2 * X).reshape(V, 4, 3)]
    nrhs = c.get("nrhs", 1)
    if V * nrhs > 2.2e6:  # over about twenty seconds
        return None
    return _solution(c, dims, c["kappa"], seed, nrhs, c["what"] == "laplace")


def _exact_apply(c, dims, seed):
    V, nrhs = inputs.volume(dims), c["nrhs"]
    if V * nrhs > 8e6:
        return None
    U = _grid(_links(c, dims, seed), dims, (4, 3, 3))
    x = _apply_input(c, seed)
    kappa = c["kappa"]
    if c["kind"] == "full":
        D = _operator(U, kappa)
        g = _grid(x, dims, (4, 3))
        parities = [0, 1]
    else:
        par = 0 if c["kind"] == "even" else 1
        keep = _parity_mask(dims, par)
        full = torch.zeros(nrhs, V, 4, 3, dtype=torch.complex128, device="cuda")
        full[:, keep] = x.reshape(nrhs, -1, 4, 3)
        g = _grid(full, dims, (4, 3))
        D = lambda p, sign=1: p - kappa * kappa * _hopping(U, _hopping(U, p, sign), sign)  # noqa: E731
        parities = [par]
    y = {"apply": lambda: D(g), "norm": lambda: D(g), "dag": lambda: D(g, -1), "normal": lambda: D(D(g), -1)}[c["op"]]()
    y = y.reshape(nrhs, V, 12)
    norm = y.abs().square().sum((1, 2))
    if c["prec"] == "df64":
        own = y if c["kind"] == "full" else y[:, _parity_mask(dims, parities[0])]
        own = own.reshape((nrhs, -1, 4, 3) if nrhs > 1 else (-1, 4, 3))
    else:
        rows, scales = [], []
        for r in range(nrhs):
            for par in parities:
                v = torch.view_as_real(y[r, _parity_mask(dims, par)]).reshape(-1, 24)
                if c["prec"] in ("f16", "bf16"):
                    top = v.abs().amax(1)
                    scales.append(top)
                    v = v / top[:, None]
                k = {"f64": 2, "f32": 4}.get(c["prec"], 8)  # numbers of one site side by side in a plane
                rows.append(v.reshape(-1, 24 // k, k).transpose(0, 1).reshape(-1))
        own = torch.cat(rows)
        if scales:
            own = [own.view(len(rows), -1), torch.stack(scales)]
    return [norm.cpu().numpy(), own] if c["op"] == "norm" else own


def _parity_mask(dims, par):
    i = torch.arange(inputs.volume(dims), device="cuda")
    x, q = i % dims[0], i // dims[0]
    y, q = q % dims[1], q // dims[1]
    return (x + y + q % dims[2] + q // dims[2]) % 2 == par
