"""The calls whose time matters to a user of the Wilson library, at the sizes they are made at.

A lattice QCD program creates one gauge object per configuration and keeps it; with it
it converts fields, applies the hopping term and the (clover) Wilson matrix in the
precision of its choice, forms dot products and solves D x = b.  Every case is one such
call, or for field conversion the few calls that go together, through the Python binding
of the C ABI.  Sizes are those of workloads.py, the tests and the benchmark, and a ragged
one whose half volume fills no block, tile or wave evenly.
"""
from __future__ import annotations

import math

import torch

from paper_1811_00893_gb300 import wilson
from paper_1811_00893_gb300.workloads import BATCH_SHAPES, BC_PPPA

PRECS = {"f64": wilson.WL_F64, "f32": wilson.WL_F32, "f16": wilson.WL_F16}
SPINOR_BYTES = {"f64": 192, "f32": 96, "f16": 52}  # one site, one right-hand side
LINK_BYTES = {"f64": 1152, "f32": 576, "f16": 288}  # the eight links of one output site
KAPPA = {"haar": 0.12, "smooth": 0.124}


def _case(name, op, dims, prec, nrhs=1, links="smooth", eo=1, dagger=0, r12=False, clover=False):
    c = {"op": op, "Lx": dims[0], "Ly": dims[1], "Lz": dims[2], "Lt": dims[3], "prec": prec, "nrhs": nrhs,
         "links": links, "eo": eo, "dagger": dagger, "r12": r12, "clover": clover}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one hopping application on a test-sized lattice, where the launch counts
        _case("dslash_f32_8x8x8x8", "dslash", (8, 8, 8, 8), "f32", links="haar"),
        # the paper's protocol: the hopping term, one right-hand side, a production-sized lattice
        _case("dslash_f32_32x32x32x64", "dslash", (32, 32, 32, 64), "f32"),
        # the even-odd matrix in 16-bit storage on the largest lattice of the workloads
        _case("mult_f16_48x48x48x96", "mult", (48, 48, 48, 96), "f16"),
        # a propagator's twelve spin-colour sources through one matrix application
        _case("mult_f32_24x24x24x48_rhs12", "mult", (24, 24, 24, 48), "f32", nrhs=12, links="haar"),
        # the clover matrix (improved action): its even-odd form
        _case("mult_f32_clover_32x32x32x64", "mult", (32, 32, 32, 64), "f32", clover=True),
        # the full matrix's adjoint in double precision (residual checks, normal equations), ragged extents
        _case("mult_f64_full_dag_20x18x14x30", "mult", (20, 18, 14, 30), "f64", links="haar", eo=0, dagger=1),
        # the even-odd adjoint with compressed links
        _case("mult_f32_r12_dag_24x24x24x48", "mult", (24, 24, 24, 48), "f32", dagger=1, r12=True),
        # sources in, dot products, results out: what surrounds the operator in a user's own solver
        _case("fields_f32_24x24x24x48_rhs12", "fields", (24, 24, 24, 48), "f32", nrhs=12, links="haar"),
        # plain double-precision BiCGStab on a small lattice, no preconditioning
        _case("solve_f64_full_8x8x8x8", "solve", (8, 8, 8, 8), "f64", links="haar", eo=0),
        # the headline: mixed-precision solve of one source
        _case("solve_f32_32x32x32x64", "solve", (32, 32, 32, 64), "f32"),
        # twelve sources solved together
        _case("solve_f32_24x24x24x48_rhs12", "solve", (24, 24, 24, 48), "f32", nrhs=12, links="haar"),
        # sixteen lattices of uneven size with one to eight sources each, solved as one batch
        {"name": "batch_f32_16", "op": "batch", "nlat": 16, "pick": 5005, "prec": "f32", "links": "haar"},
    ]


def draw(rng):
    op = rng.choice(["dslash", "dslash", "mult", "mult", "mult", "fields", "solve", "solve", "batch"])
    if op == "batch":
        return {"op": "batch", "nlat": rng.randint(2, 12), "pick": rng.randrange(1 << 20), "prec": rng.choice(["f32", "f32", "f16"]),
                "links": "haar"}
    prec = rng.choice(["f32", "f32", "f32", "f16", "f64"])
    # site-rhs pairs over the listed cases' range (their logarithm uniform), bounded by the largest call of the kind
    most = {"solve": {"f32": 1.5e6, "f16": 1.5e6, "f64": 2.0e5}, "fields": {"f32": 4.0e6, "f16": 4.0e6, "f64": 2.0e6}}.get(
        op, {"f32": 3.0e6, "f16": 6.0e6, "f64": 1.2e6})[prec]
    work = math.exp(rng.uniform(math.log(4096), math.log(most)))
    nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8, 12])
    while nrhs > 1 and work / nrhs < 2000:
        nrhs //= 2
    side = (work / nrhs) ** 0.25
    dims = [max(4, 2 * round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(4)]
    while dims[0] * dims[1] * dims[2] * dims[3] * nrhs > most:
        dims[dims.index(max(dims))] -= 2
    return _case(None, op, dims, prec, nrhs=nrhs, links=rng.choice(["haar", "smooth"]),
                 eo=rng.choice([0, 1, 1]), dagger=0 if op in ("solve", "fields") else rng.choice([0, 0, 1]),
                 r12=op in ("dslash", "mult") and prec != "f64" and rng.random() < 0.2,
                 clover=op in ("mult", "solve") and rng.random() < 0.25)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _randn(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")


def _unit_rows(a, b):
    """SU(3) matrices from two rows: Gram-Schmidt, then the third as conj(a x b)."""
    a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
    for _ in range(2):
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2)


def _gauge_field(V, links, seed):
    """(V, 4, 3, 3): Haar SU(3) links, or smooth ones near 1 (Gaussian algebra elements of width 0.3)."""
    U = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
    step = 1 << 20
    for at in range(0, V, step):
        n = min(step, V - at)
        if links == "haar":
            z = torch.view_as_complex(_randn((n, 4, 2, 3, 2), seed * 64 + at // step))
            a, b = z[:, :, 0], z[:, :, 1]
        else:  # the first two rows of 1 + i 0.3 A - (0.3 A)^2 / 2, A = sum of omega_a lambda_a / 2
            w = 0.15 * _randn((8, n, 4), seed * 64 + at // step)
            d8 = w[7] / math.sqrt(3)
            A = torch.stack([torch.stack([torch.complex(w[2] + d8, 0 * d8), torch.complex(w[0], -w[1]), torch.complex(w[3], -w[4])], -1),
                             torch.stack([torch.complex(w[0], w[1]), torch.complex(d8 - w[2], 0 * d8), torch.complex(w[5], -w[6])], -1),
                             torch.stack([torch.complex(w[3], w[4]), torch.complex(w[5], w[6]), torch.complex(-2 * d8, 0 * d8)], -1)], -2)
            E = torch.eye(3, dtype=A.dtype, device=A.device) + 1j * A - 0.5 * (A[..., :, :, None] * A[..., None, :, :]).sum(-2)
            a, b = E[..., 0, :], E[..., 1, :]
        U[at:at + n] = _unit_rows(a, b)
    return U


def _sources(nrhs, V, seed):
    return torch.view_as_complex(_randn((nrhs, V, 4, 3, 2), seed))


def _clover_field(V, seed):
    """Hermitian blocks, well conditioned once 1 is added (0.1 times Gaussians of unit total width)."""
    Z = torch.view_as_complex(_randn((V, 2, 6, 6, 2), seed)) / math.sqrt(12.0)
    return 0.05 * (Z + Z.conj().transpose(-1, -2))


def _dims(case):
    return case["Lx"], case["Ly"], case["Lz"], case["Lt"]


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _members(case):
    """Extents, sources and kappa of a batch's lattices."""
    g = torch.Generator()
    g.manual_seed(case["pick"])
    r = torch.rand((case["nlat"], 3), generator=g, dtype=torch.float64).tolist()
    return [(BATCH_SHAPES[int(a * len(BATCH_SHAPES))], 1 + int(8 * b), 0.11 + 0.014 * c) for a, b, c in r]


def _systems(case):
    """(dims, nrhs, kappa) of every lattice of a case."""
    if case["op"] == "batch":
        return _members(case)
    return [(_dims(case), case["nrhs"], KAPPA[case["links"]])]


def _inputs(case, seed):
    """Canonical links, sources and clover field of every lattice of a case."""
    for l, (dims, nrhs, kappa) in enumerate(_systems(case)):
        V, at = _volume(dims), 8 * (seed * 16 + l)
        yield (dims, nrhs, kappa, _gauge_field(V, case["links"], at + 1), _sources(nrhs, V, at + 2),
               _clover_field(V, at + 3) if case.get("clover") else None)


def _solve_params(case):
    return wilson.solve_params(tol=1e-10, eo=bool(case.get("eo", 1)), inner=PRECS[case["prec"]],
                               delta=0.003 if case["prec"] == "f16" else 0.0)


def _to_internal(g, psi, prec, nrhs, parity):
    """Internal field of canonical psi: its sites of one parity, or [even | odd] per right-hand side (None)."""
    p = PRECS[prec]
    if parity is not None:
        f = g.field(p, nrhs)
        wilson.wl_field_to_internal(g.handle, f, psi, parity, p, nrhs)
        return f
    f = g.field(p, nrhs, 2).reshape(nrhs, 2, -1)
    for r in range(nrhs):
        for parity in (0, 1):
            wilson.wl_field_to_internal(g.handle, f[r, parity], psi[r], parity, p, 1)
    return f


def prepare(case, seed):
    prec = case["prec"]
    s = {"op": case["op"], "prec": prec, "parts": []}
    for dims, nrhs, kappa, U, psi, F in _inputs(case, seed):
        g = wilson.Gauge(dims, kappa, U, precs=("f64", prec), bc=BC_PPPA, r12=bool(case.get("r12")))
        if F is not None:
            wilson.wl_clover_set(g.handle, F)
        part = {"g": g, "nrhs": nrhs}
        if case["op"] in ("solve", "batch"):
            part["b"], part["x"] = psi, torch.zeros_like(psi)
        elif case["op"] == "fields":
            part["psi"], part["back"] = psi, torch.zeros_like(psi)
            part["even"], part["odd"] = g.field(prec, nrhs), g.field(prec, nrhs)
            part["dots"] = torch.zeros((2, nrhs, 3), dtype=torch.float64, device="cuda")
        else:
            full = case["op"] == "mult" and not case["eo"]
            part["in"] = _to_internal(g, psi, prec, nrhs, None if full else 1 if case["op"] == "dslash" else 0)
            part["out"] = torch.empty_like(part["in"])
            part["full"], part["dagger"] = full, case["dagger"]
        s["parts"].append(part)
        del U
    if case["op"] in ("solve", "batch"):
        s["params"] = _solve_params(case)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _values(field, prec, nrhs):
    """An internal field's numbers: 16-bit fields are words and one FP32 norm per site."""
    if prec == "f64":
        return field.reshape(-1).view(torch.float64)
    if prec == "f32":
        return field.reshape(-1).view(torch.float32)
    rows = field.reshape(field.shape[0] * field.shape[1] if field.dim() == 3 else nrhs, -1)  # one half field each
    n = rows.shape[1] // 52 * 48
    return [rows[:, :n].view(torch.float16), rows[:, n:].view(torch.float32)]


def run(state):
    op, prec = state["op"], PRECS[state["prec"]]
    if op == "batch":
        parts = state["parts"]
        wilson.wilson_solve_batch([p["g"].handle for p in parts], [p["x"] for p in parts], [p["b"] for p in parts],
                                  [p["nrhs"] for p in parts], state["params"])
        return [p["x"] for p in parts]
    p = state["parts"][0]
    g, nrhs = p["g"].handle, p["nrhs"]
    if op == "solve":
        wilson.wilson_solve(g, p["x"], p["b"], nrhs, state["params"])
        return p["x"]
    if op == "fields":
        wilson.wl_field_to_internal(g, p["even"], p["psi"], 0, prec, nrhs)
        wilson.wl_field_to_internal(g, p["odd"], p["psi"], 1, prec, nrhs)
        wilson.wl_cdot(g, p["dots"][0], p["even"], p["even"], prec, nrhs)
        wilson.wl_cdot(g, p["dots"][1], p["even"], p["odd"], prec, nrhs)
        wilson.wl_field_to_canonical(g, p["back"], p["even"], 0, prec, nrhs)
        wilson.wl_field_to_canonical(g, p["back"], p["odd"], 1, prec, nrhs)
        return [p["dots"], p["back"]]
    if op == "dslash":
        wilson.wilson_dslash(g, p["out"], p["in"], 0, p["dagger"], prec, nrhs)
    else:
        wilson.wilson_mult(g, p["out"], p["in"], 0 if p["full"] else 1, p["dagger"], prec, nrhs)
    return _values(p["out"], state["prec"], nrhs)


def work(case):
    """Each link, clover matrix, input and output moved once, in the case's storage format;
    1320 flop per hopping application of a site, the two of one iteration at least for a solve."""
    total_bytes = total_flops = 0.0
    for dims, nrhs, _ in _systems(case):
        V, prec = _volume(dims), case["prec"]
        link, spinor = LINK_BYTES[prec] * (2 / 3 if case.get("r12") else 1.0), SPINOR_BYTES[prec]
        sites = V / 2
        if case["op"] == "fields":
            total_bytes += V * nrhs * (192 + 192)
            total_flops += V * nrhs * 24 * 8
            continue
        if case["op"] == "dslash":
            total_bytes += sites * (link + 2 * spinor * nrhs)
            total_flops += sites * nrhs * 1320
            continue
        if case["op"] == "mult":
            total_bytes += V * link + (V if not case["eo"] else sites) * 2 * spinor * nrhs
            total_flops += V * nrhs * 1320
        else:
            total_bytes += V * link + V * nrhs * 2 * 192
            total_flops += 2 * V * nrhs * 1320
        if case.get("clover"):
            total_bytes += V * (LINK_BYTES[prec] / 2)
            total_flops += V * nrhs * 504
    return {"bytes": total_bytes, "flops": total_flops}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

# (1 + S gamma_mu): gamma_mu's only entry in each row, as (column, value), DeGrand-Rossi basis
_GAMMA = [
    [(3, 1j), (2, 1j), (1, -1j), (0, -1j)],
    [(3, -1), (2, 1), (1, 1), (0, -1)],
    [(2, 1j), (3, -1j), (0, -1j), (1, 1j)],
    [(2, 1), (3, 1), (0, 1), (1, 1)],
]


def _gamma(mu, q):
    return torch.stack([v * q[..., c, :] for c, v in _GAMMA[mu]], dim=-2)


class _Wilson:
    """H, D and the even-odd matrix on fields (nrhs, Lt, Lz, Ly, Lx, 4, 3) of complex doubles."""

    def __init__(self, dims, kappa, U, F):
        Lx, Ly, Lz, Lt = dims
        self.dims, self.kappa = dims, kappa
        self.U = U.reshape(Lt, Lz, Ly, Lx, 4, 3, 3)
        n = [torch.arange(L, device=U.device) for L in (Lt, Lz, Ly, Lx)]
        parity = n[0][:, None, None, None] + n[1][:, None, None] + n[2][:, None] + n[3]
        self.odd = (parity % 2 == 1)
        self.A = None if F is None else (F + torch.eye(6, dtype=F.dtype, device=F.device)).reshape(Lt, Lz, Ly, Lx, 2, 6, 6)
        self.Ainv = None if F is None else torch.linalg.inv(self.A)

    def mask(self, psi, odd):
        return psi * (self.odd if odd else ~self.odd)[..., None, None]

    def block(self, M, psi):
        if M is None:
            return psi
        q = psi.reshape(*psi.shape[:-2], 2, 6)
        return torch.stack([(M[..., i, :] * q).sum(-1) for i in range(6)], dim=-1).reshape(psi.shape)

    def hop(self, psi, dagger=0):
        out = torch.zeros_like(psi)
        for mu in range(4):
            d = psi.dim() - 3 - mu
            L, ph, S = self.dims[mu], BC_PPPA[mu], (1 if dagger else -1)
            U = self.U[..., mu, :, :]
            q = psi + S * _gamma(mu, psi)  # forward: (1 -+ gamma) psi(x + mu)
            q = torch.roll(q, -1, d)
            if ph != 1:
                q.select(d, L - 1).mul_(ph)
            out += torch.stack([(U[..., None, a, :] * q).sum(-1) for a in range(3)], dim=-1)
            q = psi - S * _gamma(mu, psi)  # backward: U(x - mu)^dag
            q = torch.stack([(U[..., None, :, a].conj() * q).sum(-1) for a in range(3)], dim=-1)
            q = torch.roll(q, 1, d)
            if ph != 1:
                q.select(d, 0).mul_(ph)
            out += q
        return out

    def full(self, psi, dagger=0):
        return self.block(self.A, psi) - self.kappa * self.hop(psi, dagger)

    def even(self, psi, dagger=0):
        """The Schur complement of the full matrix on fields that live on the even sites."""
        t = self.mask(self.block(self.Ainv, self.hop(psi, dagger)), True)
        return self.block(self.A, psi) - self.kappa ** 2 * self.mask(self.hop(t, dagger), False)

    def solve(self, b):
        """BiCGStab on the full matrix to 1e-13, one right-hand side at a time."""
        x, r = torch.zeros_like(b), b.clone()
        rh, goal = r.clone(), 1e-13 * float(torch.linalg.vector_norm(b))
        rho = torch.vdot(rh.reshape(-1), r.reshape(-1))
        p = r.clone()
        for _ in range(400):
            v = self.full(p)
            alpha = rho / torch.vdot(rh.reshape(-1), v.reshape(-1))
            s = r - alpha * v
            t = self.full(s)
            omega = torch.vdot(t.reshape(-1), s.reshape(-1)) / torch.vdot(t.reshape(-1), t.reshape(-1))
            x += alpha * p + omega * s
            r = s - omega * t
            if float(torch.linalg.vector_norm(r)) <= goal:
                break
            new = torch.vdot(rh.reshape(-1), r.reshape(-1))
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        return x


def _layout(M, psi, prec, parities):
    """psi's sites in the order and planes of internal fields of the given parities."""
    words, norms = [], []
    for r in range(psi.shape[0]):
        for odd in parities:
            v = psi[r][M.odd if odd else ~M.odd].reshape(-1, 12)  # site order within a parity is the half index
            if prec == "f64":
                words.append(v.t())
            elif prec == "f32":
                words.append(v.reshape(-1, 6, 2).transpose(0, 1))
            else:
                m = torch.view_as_real(v).abs().amax((-2, -1))
                words.append((v / m[:, None]).reshape(-1, 3, 4).transpose(0, 1))
                norms.append(m)
    flat = [torch.view_as_real(w.contiguous()).reshape(-1) for w in words]
    return torch.cat(flat) if prec != "f16" else [torch.stack(flat), torch.stack(norms)]


def exact(case, seed):
    out = []
    for dims, nrhs, kappa, U, psi, F in _inputs(case, seed):
        M = _Wilson(dims, kappa, U, F)
        q = psi.reshape(nrhs, dims[3], dims[2], dims[1], dims[0], 4, 3)
        if case["op"] in ("solve", "batch"):
            out.append(torch.cat([M.solve(q[r:r + 1]) for r in range(nrhs)]).reshape(psi.shape))
        elif case["op"] == "fields":
            # the dot product pairs the even and the odd site of each half index
            ev = torch.stack([q[r][~M.odd].reshape(-1) for r in range(nrhs)])
            od = torch.stack([q[r][M.odd].reshape(-1) for r in range(nrhs)])
            ee, oo = (ev.abs() ** 2).sum(-1), (od.abs() ** 2).sum(-1)
            eo = (ev.conj() * od).sum(-1)
            return [torch.stack([torch.stack([ee, 0 * ee, ee], -1), torch.stack([eo.real, eo.imag, oo], -1)]), psi]
        elif case["op"] == "dslash":
            q = M.mask(q, True)
            return _layout(M, torch.cat([M.hop(q[r:r + 1], case["dagger"]) for r in range(nrhs)]), case["prec"], (0,))
        elif case["eo"]:
            q = M.mask(q, False)
            return _layout(M, torch.cat([M.even(q[r:r + 1], case["dagger"]) for r in range(nrhs)]), case["prec"], (0,))
        else:
            return _layout(M, torch.cat([M.full(q[r:r + 1], case["dagger"]) for r in range(nrhs)]), case["prec"], (0, 1))
    return out if case["op"] == "batch" else out[0]
