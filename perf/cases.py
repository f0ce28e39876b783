"""What a program that uses this framework has it do, as cases to be timed.

Each case is one pass through the public entry points (binding.py, autograd.py)
on one lattice or a few: the operator on caller's spinors and on resident
fields, solves, the gradient through a solve, the fermion force, and what a
molecular-dynamics step does with a new gauge field.  Lattices, Schwarz blocks
and masses are those of this repository's workloads, tests and benchmark.

Results are handed back in the precision they were asked for in: an FP32
operator's as complex64, a 16-bit one's as 16-bit (re, im) pairs, the others as
they come (complex128 / float64).
"""
from __future__ import annotations

import math

import torch

from paper_1109_4279_gb300 import autograd
from paper_1109_4279_gb300 import binding as B

AP = (-1.0, 1.0, 1.0, 1.0)  # antiperiodic time
UNEVEN = {(8, 8, 8, 8): (4, 4, 2, 2), (16, 8, 8, 8): (4, 4, 4, 4), (24, 12, 12, 12): (4, 6, 2, 2),
          (32, 16, 16, 16): (4, 4, 4, 4)}


def _text(v):
    return "x".join(str(k) for k in v)


def _dims(t):
    return tuple(int(k) for k in t.split("x"))


def _case(name, kind, dims, block, **kw):
    return dict({"name": name, "kind": kind, "dims": _text(dims), "block": _text(block), "m0": 0.0, "csw": 1.5,
                 "eps": 0.5}, **kw)


def listed():
    return [
        # the smallest call: a program that drives its own iteration on a toy lattice; latency and launches
        _case("apply f64 4^4", "apply", (4, 4, 4, 4), (2, 2, 2, 2), prec="f64", dagger=False, nrhs=1, m0=0.1, csw=1.0,
              eps=0.3),
        # a caller's own solver on an ordinary lattice: D^+ at double accuracy on the FP32 units
        _case("apply df64 D+ 16^3x32", "apply", (32, 16, 16, 16), (4, 4, 4, 4), prec="df64", dagger=True, nrhs=1),
        # single precision on blocks that are no power of two, two right-hand sides
        _case("apply f32 12^3x24 x2", "apply", (24, 12, 12, 12), (4, 6, 2, 2), prec="f32", dagger=False, nrhs=2),
        # a caller's iteration on resident fields (D, D^+ in turn), the largest lattice: HBM traffic
        _case("resident f32 32^3x64", "resident", (64, 32, 32, 32), (4, 4, 4, 4), prec="f32", applies=4, nrhs=1,
              m0=-0.05),
        # the same for the 12 spin-colour right-hand sides of one propagator, 16-bit storage
        _case("resident f16 24^3x48 x12", "resident", (48, 24, 24, 24), (8, 4, 4, 4), prec="f16", applies=2, nrhs=12),
        # a small solve with the library's default parameters: latency
        _case("solve default 8^3x16", "solve", (16, 8, 8, 8), (4, 4, 4, 4), nrhs=1, sap_prec="f32", outer_prec="f64",
              m0=-0.05),
        # the benchmarked solve: one Gaussian right-hand side on the largest lattice
        _case("solve f16 32^3x64", "solve", (64, 32, 32, 32), (8, 4, 4, 4), nrhs=1, sap_prec="f16", outer_prec="df64",
              m0=-0.05),
        # a propagator: 12 point sources in one call
        _case("propagator 24^3x48", "propagator", (48, 24, 24, 24), (8, 4, 4, 4), sap_prec="f16", outer_prec="df64"),
        # ten lattices of four sizes in one call, one right-hand side each
        _case("uneven batch", "uneven", (32, 16, 16, 16), (4, 4, 4, 4), copies=1, sap_prec="f16", outer_prec="df64"),
        # forward and backward through a solve: adjoint solve and force
        _case("gradient 16^3x32", "gradient", (32, 16, 16, 16), (4, 4, 4, 4), sap_prec="f16", outer_prec="df64"),
        # the fermion force of given solutions
        _case("force 24^3x48", "force", (48, 24, 24, 24), (4, 4, 4, 4)),
        # the gauge half of a molecular-dynamics step: gauge force, link update, the new links loaded with their
        # clover term, and the pseudofermion's D^+ on them
        _case("md step 16^3x32", "md", (32, 16, 16, 16), (4, 4, 4, 4)),
    ]


BLOCKS = ((2, 2, 2, 2), (4, 2, 2, 4), (4, 4, 2, 2), (4, 6, 2, 2), (4, 4, 4, 4), (8, 4, 4, 4))


def _draw_lattice(rng, least, most, blocks):
    """Block and extents (even block counts), the volume spread over its logarithm."""
    block = rng.choice(blocks)
    vb = math.prod(block)
    want = math.exp(rng.uniform(math.log(max(least, 16 * vb)), math.log(most)))
    best = None
    for _ in range(40):
        dims = tuple(b * 2 * rng.randint(1, max(1, 32 // b)) for b in block)
        off = abs(math.log(math.prod(dims) / want)) + (10.0 if math.prod(dims) > most else 0.0)
        if best is None or off < best[0]:
            best = (off, dims)
    if math.prod(best[1]) > most:  # the smallest lattice of these blocks
        return tuple(2 * b for b in block), block
    return best[1], block


def draw(rng):
    kind = rng.choice(("apply", "apply", "resident", "resident", "solve", "solve", "propagator", "uneven", "gradient",
                       "force", "md"))
    m0 = rng.choice((-0.05, 0.0, 0.1))
    mixed = dict(sap_prec=rng.choice(("f16", "f16", "f32", "bf16")), outer_prec="df64")
    small = tuple(b for b in BLOCKS if math.prod(b) <= 256)  # FP32 block fields of larger blocks do not fit
    if kind == "apply":
        nrhs = rng.choice((1, 1, 2, 3))
        dims, block = _draw_lattice(rng, 256, 1000000 // nrhs, BLOCKS)
        c = _case("", kind, dims, block, prec=rng.choice(("f64", "df64", "f32", "f16", "bf16")),
                  dagger=rng.random() < 0.5, nrhs=nrhs)
    elif kind == "resident":
        nrhs = rng.choice((1, 1, 2, 5, 12))
        dims, block = _draw_lattice(rng, 4096, 2097152 // nrhs if nrhs < 12 else 663552, BLOCKS)
        c = _case("", kind, dims, block, prec=rng.choice(("f64", "f32", "f16", "bf16")), applies=rng.randint(1, 4),
                  nrhs=nrhs)
    elif kind == "solve":
        opts = dict(sap_prec="f32", outer_prec="f64") if rng.random() < 0.3 else mixed
        dims, block = _draw_lattice(rng, 4096, 600000, small if opts["sap_prec"] == "f32" else BLOCKS[2:])
        c = _case("", kind, dims, block, nrhs=rng.choice((1, 1, 1, 2)), **opts)
    elif kind == "propagator":
        dims, block = _draw_lattice(rng, 4096, 150000, BLOCKS[2:])
        c = _case("", kind, dims, block, **dict(mixed, sap_prec="f16"))
    elif kind == "uneven":
        c = _case("", kind, (32, 16, 16, 16), (4, 4, 4, 4), copies=rng.randint(1, 3), **dict(mixed, sap_prec="f16"))
    elif kind == "gradient":
        dims, block = _draw_lattice(rng, 4096, 300000, BLOCKS[2:])
        c = _case("", kind, dims, block, **dict(mixed, sap_prec="f16"))
    else:
        dims, block = _draw_lattice(rng, 4096, 700000 if kind == "force" else 300000, BLOCKS)
        c = _case("", kind, dims, block)
    c["m0"], c["eps"] = m0, round(rng.uniform(0.3, 0.5), 3)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gell_mann(dev):
    g = torch.zeros((8, 3, 3), dtype=torch.complex128)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        g[a, i, j] = g[a, j, i] = 1
        g[a + 1, i, j], g[a + 1, j, i] = -1j, 1j
    g[2, 0, 0], g[2, 1, 1] = 1, -1
    g[7] = torch.diag(torch.tensor([1, 1, -2], dtype=torch.complex128)) / math.sqrt(3.0)
    return g.to(dev)


def _unitary(m):
    """Rows 0 and 1 orthonormalised, row 2 = conj(row 0 x row 1): SU(3)."""
    r0 = m[..., 0, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = m[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1).conj()
    return torch.stack((r0, r1, r2), dim=-2).contiguous()


def _links(V, eps, gen):
    """Random links near exp(i eps sum_a g_a lambda_a / 2), g_a ~ N(0, 1)."""
    dev = gen.device
    lam = (_gell_mann(dev) / 2).reshape(8, 9)
    one = torch.eye(3, dtype=torch.complex128, device=dev)
    out = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device=dev)
    step = 1 << 18
    for s in range(0, V, step):
        n = min(step, V - s)
        g = torch.randn((n * 4, 8), dtype=torch.float64, device=dev, generator=gen)
        h = (1j * eps * (g.to(torch.complex128) @ lam)).reshape(-1, 3, 3)
        h2 = (h.unsqueeze(-1) * h.unsqueeze(-3)).sum(-2)  # h h, and exp to third order: Gram-Schmidt does the rest
        h3 = (h2.unsqueeze(-1) * h.unsqueeze(-3)).sum(-2)
        out[s:s + n] = _unitary(one + h + h2 / 2 + h3 / 6).reshape(n, 4, 3, 3)
    return out


def _spinor(V, gen, n=None):
    shape = (V, 4, 3, 2) if n is None else (n, V, 4, 3, 2)
    return torch.view_as_complex(torch.randn(shape, dtype=torch.float64, device=gen.device, generator=gen))


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 7919 + 1)
    return gen


def _fields(case, gen, dims=None):
    dims = dims or _dims(case["dims"])
    return dims, math.prod(dims), _links(math.prod(dims), case["eps"], gen)


def _lattice(case, U, dims=None, block=None):
    lat = B.Lattice(dims or _dims(case["dims"]), block or _dims(case["block"]), case["m0"], case["csw"], AP)
    lat.load_gauge(U)
    return lat


def _uneven_dims(case):
    return ([(8, 8, 8, 8)] * 2 + [(16, 8, 8, 8)] * 2 + [(24, 12, 12, 12)] * 3 + [(32, 16, 16, 16)] * 3) * case["copies"]


def _solver(case):
    return dict(tol=1e-10, sap_prec=case["sap_prec"], outer_prec=case["outer_prec"])


def _sources(V, gen):
    """12 spin-colour point sources at one site."""
    site = int(torch.randint(0, V, (1,), device=gen.device, generator=gen))
    b = torch.zeros((12, V, 4, 3), dtype=torch.complex128, device=gen.device)
    for s in range(4):
        for c in range(3):
            b[s * 3 + c, site, s, c] = 1.0
    return b


def _inputs(case, seed):
    """The tensors of a case (the lattice handle is made from U)."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "uneven":
        parts = []
        for dims in _uneven_dims(case):
            _, V, U = _fields(case, gen, dims)
            parts.append((dims, U, _spinor(V, gen)))
        return {"parts": parts}
    dims, V, U = _fields(case, gen)
    d = {"U": U}
    if kind in ("apply", "resident", "solve"):
        d["psi"] = _spinor(V, gen, case["nrhs"] if case["nrhs"] > 1 else None)
    elif kind == "propagator":
        d["psi"] = _sources(V, gen)
    elif kind == "gradient":
        d["psi"], d["g"] = _spinor(V, gen), _spinor(V, gen)
    elif kind == "force":
        d["x"], d["y"] = _spinor(V, gen), _spinor(V, gen)
    elif kind == "md":
        d["psi"] = _spinor(V, gen)
        d["pi"] = torch.randn((V, 4, 8), dtype=torch.float64, device=gen.device, generator=gen)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "uneven":
        st["lats"] = [_lattice(case, U, dims, UNEVEN[dims]) for dims, U, _ in d["parts"]]
        st["b"] = [b for _, _, b in d["parts"]]
        return st
    st["lat"] = _lattice(case, d["U"])
    if kind == "resident":
        ctx = st["lat"].ctx
        st["fields"] = [B.qcd_field_create_n(ctx, case["prec"], case["nrhs"]) for _ in range(3)]
        B.qcd_field_import(ctx, st["fields"][0], d["psi"])
        st["out"] = torch.empty_like(d["psi"])
        st["free"] = _Fields(st["fields"], st["lat"])
        return st
    if kind == "md":
        st["U"] = d["U"]
    st.update({k: v for k, v in d.items() if k != "U"})
    return st


class _Fields:
    """Frees resident fields before their lattice goes."""

    def __init__(self, fields, lat):
        self.fields, self.lat = fields, lat

    def __del__(self):
        for f in self.fields:
            B.qcd_field_free(f)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _as_asked(out, prec):
    if prec == "f32":
        return out.to(torch.complex64)
    if prec in ("f16", "bf16"):
        return torch.view_as_real(out).to(torch.float16 if prec == "f16" else torch.bfloat16)
    return out


BETA, STEP = 5.29, 0.02


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        return _as_asked(state["lat"].apply_D(state["psi"], dagger=case["dagger"], prec=case["prec"]), case["prec"])
    if kind == "resident":
        ctx, f = state["lat"].ctx, state["fields"]
        src = f[0]
        for k in range(case["applies"]):
            dst = f[1 + k % 2]
            B.qcd_apply_D_field(ctx, src, dst, dagger=bool(k % 2))
            src = dst
        B.qcd_field_export(ctx, src, state["out"])
        return _as_asked(state["out"], case["prec"])
    if kind in ("solve", "propagator"):
        return state["lat"].solve(state["psi"], **_solver(case))[0]
    if kind == "uneven":
        xs = [torch.zeros_like(b) for b in state["b"]]
        B.qcd_solve_batch([lat.ctx for lat in state["lats"]], state["b"], xs, B.solver_params(**_solver(case)))
        return xs
    if kind == "gradient":
        lat = state["lat"]
        phi = state["psi"].clone().requires_grad_(True)
        theta = torch.zeros((lat.V, 4, 8), dtype=torch.float64, device=phi.device, requires_grad=True)
        x = autograd.dirac_solve(phi, theta, lat, **_solver(case))
        x.backward(state["g"])
        return x.detach(), phi.grad, theta.grad
    if kind == "force":
        F = torch.empty((state["lat"].V, 4, 8), dtype=torch.float64, device=state["x"].device)
        B.qcd_force(state["lat"].ctx, state["x"], state["y"], F)
        return F
    lat = state["lat"]
    U = state["U"].clone()
    F = torch.empty((lat.V, 4, 8), dtype=torch.float64, device=U.device)
    B.qcd_gauge_force(lat.ctx, U, BETA, F)
    B.qcd_update_links(lat.ctx, U, state["pi"], STEP)
    lat.load_gauge(U)
    return F, U, lat.apply_D(state["psi"], dagger=True)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
WIDTH = {"f64": 8, "df64": 8, "f32": 4, "f16": 2, "bf16": 2}


def _operator_bytes(prec):
    """Links (two rows below 64 bits) and clover of a site in a storage precision."""
    w = WIDTH[prec]
    return (72 if w == 8 else 48) * w + 72 * w + (4 if w == 2 else 0)


def work(case):
    kind = case["kind"]
    V = math.prod(_dims(case["dims"]))
    hop = 1824.0  # flops of one D per site
    if kind == "apply":  # the caller's spinors in and out, links and clover once
        return {"bytes": V * (384.0 * case["nrhs"] + _operator_bytes(case["prec"])), "flops": hop * V * case["nrhs"]}
    if kind == "resident":
        per = 48 * WIDTH[case["prec"]] + (8 if WIDTH[case["prec"]] == 2 else 0)
        out = 192.0 + {"f64": 0, "f32": 96 + 192, "f16": 48 + 192, "bf16": 48 + 192}[case["prec"]]
        return {"bytes": V * (case["applies"] * (per * case["nrhs"] + _operator_bytes(case["prec"])) +
                              (per / 2 + out) * case["nrhs"]), "flops": case["applies"] * hop * V * case["nrhs"]}
    # a solve of these lattices takes about six iterations of four SAP cycles (four MR steps each) and one D
    solve_flops = 6 * (4 * 5 + 1) * hop
    if kind == "uneven":
        V = sum(math.prod(d) for d in _uneven_dims(case))
    if kind in ("solve", "propagator", "uneven"):
        n = {"solve": case.get("nrhs", 1), "propagator": 12, "uneven": 1}[kind]
        w = _operator_bytes(case["sap_prec"]) + _operator_bytes(case["outer_prec"])
        return {"bytes": V * (384.0 * n + w), "flops": n * V * solve_flops}
    # 3x3 complex products of 198 flops: per site and plane the four leaves' worth
    mat = 198.0
    force = 4 * 6 * 8 * mat
    if kind == "force":
        return {"bytes": V * (384.0 + 576.0 + 256.0), "flops": V * force}
    if kind == "gradient":
        w = _operator_bytes(case["sap_prec"]) + _operator_bytes(case["outer_prec"])
        return {"bytes": V * (192.0 * 4 + 256.0 + 576.0 + w), "flops": V * (2 * solve_flops + force)}
    # md: gauge force, exponential, clover term and its inverse on half the sites, one D
    flops = 4 * 13 * mat + 4 * 16 * mat + 6 * 4 * 3 * mat + 5000.0 + hop
    return {"bytes": V * (576.0 + 256.0 * 2 + 576.0 * 2 + 1152.0 + 384.0), "flops": V * flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from plain torch
# ---------------------------------------------------------------------------
def _gammas(dev):
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    g[0, 0, 2] = g[0, 1, 3] = g[0, 2, 0] = g[0, 3, 1] = -1
    pauli = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)
    for k in range(3):
        g[k + 1, :2, 2:] = -1j * pauli[k]
        g[k + 1, 2:, :2] = 1j * pauli[k]
    return g.to(dev)


class _Plain:
    """D of given links, with whole-lattice tensors (T, X, Y, Z, ...)."""

    def __init__(self, case, dims, U):
        self.dims, self.V = dims, math.prod(dims)
        self.U = U.reshape(*dims, 4, 3, 3)
        self.m0, self.csw = case["m0"], case["csw"]
        self.g = _gammas(U.device)
        self.one = torch.eye(4, dtype=torch.complex128, device=U.device)
        self.F = {}
        for m in range(4):
            for n in range(m + 1, 4):
                q = self._leaves(m, n)
                self.F[m, n] = (q - q.mH) / 8

    def link(self, mu, *steps):
        """U_mu at x + the steps (direction, +-1), the field being periodic."""
        u = self.U[..., mu, :, :]
        for d, s in steps:
            u = torch.roll(u, -s, dims=d)
        return u

    def _leaves(self, m, n):
        u = self.link
        q = u(m) @ u(n, (m, 1)) @ u(m, (n, 1)).mH @ u(n).mH
        q = q + u(n) @ u(m, (n, 1), (m, -1)).mH @ u(n, (m, -1)).mH @ u(m, (m, -1))
        q = q + u(m, (m, -1)).mH @ u(n, (m, -1), (n, -1)).mH @ u(m, (m, -1), (n, -1)) @ u(n, (n, -1))
        return q + u(n, (n, -1)).mH @ u(m, (n, -1)) @ u(n, (n, -1), (m, 1)) @ u(m).mH

    def apply(self, psi, dagger=False):
        p = psi.reshape(*self.dims, 4, 3)
        out = (4.0 + self.m0) * p
        for (m, n), F in self.F.items():
            sigma = 0.5j * (self.g[m] @ self.g[n] - self.g[n] @ self.g[m])
            out = out + 0.5j * self.csw * torch.einsum("st,...ta->...sa", sigma, torch.einsum("...ab,...sb->...sa", F, p))
        sign = -1.0 if not dagger else 1.0
        for mu in range(4):
            edge = [slice(None)] * 4
            up, down = torch.roll(p, -1, dims=mu), torch.roll(p, 1, dims=mu)
            if AP[mu] != 1.0:
                up, down = up.clone(), down.clone()
                edge[mu] = self.dims[mu] - 1
                up[tuple(edge)] *= AP[mu]
                edge[mu] = 0
                down[tuple(edge)] *= AP[mu]
            f = torch.einsum("st,...ta->...sa", self.one + sign * self.g[mu], up)
            b = torch.einsum("st,...ta->...sa", self.one - sign * self.g[mu], down)
            out = out - 0.5 * (torch.einsum("...ab,...sb->...sa", self.link(mu), f) +
                               torch.einsum("...ba,...sb->...sa", self.link(mu, (mu, -1)).conj(), b))
        return out.reshape(psi.shape)

    def solve(self, b, dagger=False):
        """Conjugate gradients on the normal equations, to rounding."""
        r = self.apply(b, not dagger)
        x, p = torch.zeros_like(b), r.clone()
        rr = (r.abs() ** 2).sum()
        stop = rr * 1e-30
        for k in range(2000):
            t = self.apply(p, dagger)
            a = rr / (t.abs() ** 2).sum()
            x = x + a * p
            r = r - a * self.apply(t, not dagger)
            new = (r.abs() ** 2).sum()
            p, rr = r + (new / rr) * p, new
            if k % 8 == 7 and bool(new < stop):
                break
        return x


def _deform(U, theta):
    """U to first order in theta: (1 + i theta_a lambda_a / 2) U."""
    t = torch.einsum("vma,aij->vmij", theta.to(torch.complex128), _gell_mann(U.device) / 2)
    return U + 1j * (t @ U)


def _exact_force(case, dims, U, x, y):
    theta = torch.zeros((math.prod(dims), 4, 8), dtype=torch.float64, device=U.device, requires_grad=True)
    s = -(y.conj() * _Plain(case, dims, _deform(U, theta)).apply(x)).sum().real
    return torch.autograd.grad(s, theta)[0]


def _exact_md(case, dims, d):
    U = d["U"]
    theta = torch.zeros((math.prod(dims), 4, 8), dtype=torch.float64, device=U.device, requires_grad=True)
    w = _deform(U, theta).reshape(*dims, 4, 3, 3)
    s = 0.0
    for m in range(4):
        for n in range(m + 1, 4):
            um, un = w[..., m, :, :], w[..., n, :, :]
            p = um @ torch.roll(un, -1, dims=m) @ torch.roll(um, -1, dims=n).mH @ un.mH
            s = s + (1.0 - torch.einsum("...ii->...", p).real / 3.0).sum()
    F = torch.autograd.grad(BETA * s, theta)[0]
    h = 1j * STEP * torch.einsum("vma,aij->vmij", d["pi"].to(torch.complex128), _gell_mann(U.device) / 2)
    e = torch.eye(3, dtype=torch.complex128, device=U.device).expand_as(h).clone()
    for k in range(24, 0, -1):  # |h| is well below 1: the series has converged
        e = torch.eye(3, dtype=torch.complex128, device=U.device) + (h @ e) / k
    U2 = e @ U
    return F, U2, _Plain(case, dims, U2).apply(d["psi"], True)


def exact(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        return None
    dims = _dims(case["dims"])
    V = math.prod(dims)
    n = case.get("nrhs", 12 if kind == "propagator" else 1)
    if kind in ("solve", "propagator", "gradient") and V * n > 150000 or V * n > 2500000 and kind != "resident":
        return None
    if kind == "resident" and V * n * case["applies"] > 17000000:
        return None
    d = _inputs(case, seed)
    if kind == "force":
        return _exact_force(case, dims, d["U"], d["x"], d["y"])
    if kind == "md":
        return _exact_md(case, dims, d)
    plain = _Plain(case, dims, d["U"])
    psi = d["psi"]
    if kind == "gradient":
        x, y = plain.solve(psi), plain.solve(d["g"], True)
        return x, y, _exact_force(case, dims, d["U"], x, y)
    rows = []
    for p in (psi if n > 1 else [psi]):
        if kind == "apply":
            p = plain.apply(p, case["dagger"])
        elif kind == "resident":
            for k in range(case["applies"]):
                p = plain.apply(p, bool(k % 2))
        else:
            p = plain.solve(p)
        rows.append(p)
    out = torch.stack(rows) if n > 1 else rows[0]
    return torch.view_as_real(out) if case.get("prec") in ("f16", "bf16") else out
