"""FP64 hopping term with fixed-point links against exact arithmetic.

The reference is the hopping term in whole numbers: links and spinors are binary64, so
multiplied by a power of two they are integers, and sums of products of integers have no
rounding.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1811_00893_gb300 import fields, wilson

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)
SHAPES = [64, 2000]  # one thread per site; six threads per site
DIMS = [(2, 2, 2, 2), (6, 2, 2, 2), (4, 4, 4, 4)]  # Vh = 8, 24 (half a tile of 16 sites, one and a half) and 128


def _ints(a, bits):
    """Real and imaginary parts of a complex array times 2^bits, as Python integers."""
    def conv(r):
        m, e = np.frexp(np.ascontiguousarray(r))
        n = np.ldexp(m, 53).astype(np.int64).astype(object)
        sh = e.astype(np.int64) - 53 + bits
        assert np.all((sh >= 0) | (r == 0)), "not a multiple of 2^-bits"
        return n * (2 ** np.maximum(sh, 0).astype(object))
    return conv(a.real), conv(a.imag)


class Exact:
    """The hopping term of one field in integers: out = (re, im) 2^-bits, and for every output
    component total = the sum of |link entry| |projected neighbour| over its 24 products."""

    def __init__(self, U, psi, dims, dagger, ubits=240, bits=200):
        shape = tuple(dims[::-1])
        U, psi = U.reshape(shape + (4, 3, 3)), psi.reshape(shape + (4, 3))
        ur, ui = _ints(U, ubits)
        pr, pi = _ints(psi, bits)
        self.bits = ubits + bits
        re = np.zeros(psi.shape, dtype=object)
        im = np.zeros(psi.shape, dtype=object)
        self.total = np.zeros(psi.shape)
        self.largest = np.zeros(psi.shape[:-2])  # largest real component of a projected neighbour
        for mu in range(4):
            ax, gam = 3 - mu, oracle.gamma(mu)
            edge = [slice(None)] * 4
            for back in (0, 1):
                sign = (1 if back else -1) * (-1 if dagger else 1)
                a = np.eye(4) + sign * gam
                # (1 +- gamma) psi, in integers and in FP64
                qr = sum(np.multiply.outer(pr[..., s, :], a[:, s].real.astype(int).astype(object)) -
                         np.multiply.outer(pi[..., s, :], a[:, s].imag.astype(int).astype(object)) for s in range(4))
                qi = sum(np.multiply.outer(pi[..., s, :], a[:, s].real.astype(int).astype(object)) +
                         np.multiply.outer(pr[..., s, :], a[:, s].imag.astype(int).astype(object)) for s in range(4))
                qr, qi = np.moveaxis(qr, -1, -2), np.moveaxis(qi, -1, -2)
                q = np.einsum("st,...tc->...sc", a, psi)
                vr, vi, v = ur[..., mu, :, :], ui[..., mu, :, :], U[..., mu, :, :]
                if back:  # U^dag psi at the neighbour, then moved here
                    vr, vi, v = np.swapaxes(vr, -1, -2), -np.swapaxes(vi, -1, -2), np.swapaxes(v, -1, -2).conj()
                else:
                    qr, qi, q = (np.roll(x, -1, ax) for x in (qr, qi, q))
                hr = (vr[..., None, :, :] * qr[..., :, None, :] - vi[..., None, :, :] * qi[..., :, None, :]).sum(-1)
                hi = (vr[..., None, :, :] * qi[..., :, None, :] + vi[..., None, :, :] * qr[..., :, None, :]).sum(-1)
                t = (np.abs(v)[..., None, :, :] * np.abs(q)[..., :, None, :]).sum(-1)
                m = np.maximum(np.abs(q.real), np.abs(q.imag)).max((-2, -1))
                if back:
                    hr, hi, t, m = (np.roll(x, 1, ax) for x in (hr, hi, t, m))
                edge[ax] = 0 if back else dims[mu] - 1
                hr[tuple(edge)] *= BC[mu]
                hi[tuple(edge)] *= BC[mu]
                edge[ax] = slice(None)
                re, im, self.total = re + hr, im + hi, self.total + t
                self.largest = np.maximum(self.largest, m)
        self.re, self.im = re.reshape(-1, 4, 3), im.reshape(-1, 4, 3)
        self.total = self.total.reshape(-1, 4, 3)
        self.largest = self.largest.reshape(-1)

    def error(self, got):
        """got - exact, real and imaginary parts (the differences are exact before they are rounded)."""
        gr, gi = _ints(got.reshape(-1, 4, 3), self.bits)
        f = np.frompyfunc(lambda n: float(n) if abs(n) < 2 ** 1000 else float("inf"), 1, 1)
        scale = 2.0 ** -self.bits
        return f(gr - self.re).astype(float) * scale, f(gi - self.im).astype(float) * scale


def _apply(g, psi, dagger):
    """The hopping term on both parities: (V, 4, 3) complex, canonical order."""
    out = torch.zeros_like(psi)
    for p in (0, 1):
        i, o = g.field("f64"), g.field("f64")
        wilson.wl_field_to_internal(g.handle, i, psi, 1 - p, wilson.WL_F64, 1)
        wilson.wilson_dslash(g.handle, o, i, p, dagger, wilson.WL_F64, 1)
        wilson.wl_field_to_canonical(g.handle, out, o, p, wilson.WL_F64, 1)
    return out[0].cpu().numpy()


def _apply_blocks(dd, psi):
    """The same on a decomposed lattice."""
    loc, out = dd.canonical(1), dd.canonical(1)
    wilson.wl_dd_scatter(dd.handle, loc, psi, 1)
    for p in (0, 1):
        di, do = dd.field("f64"), dd.field("f64")
        for k, (gk, _) in enumerate(dd.blocks):
            wilson.wl_field_to_internal(gk, di[k], loc[k], 1 - p, wilson.WL_F64, 1)
        wilson.wilson_dslash_dd(dd.handle, do, di, p, 0, wilson.WL_F64, 1)
        for k, (gk, _) in enumerate(dd.blocks):
            wilson.wl_field_to_canonical(gk, out[k], do[k], p, wilson.WL_F64, 1)
    got = torch.zeros_like(psi)
    wilson.wl_dd_gather(dd.handle, got, out, 1)
    return got[0].cpu().numpy()


def _cases(dims, links, psi):
    """(dagger, kernel's result, exact result) for links of a kind, or given ones."""
    U = fields.gauge_field(dims, links, 13) if isinstance(links, str) else links
    with wilson.Gauge(dims, 0.12, U.cuda(), precs=("f64",), bc=BC) as g:
        for dagger in (0, 1):
            yield dagger, _apply(g, psi.cuda(), dagger), Exact(U.numpy(), psi[0].numpy(), dims, dagger)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["point", "integers"])
def test_exact_on_unit_links(dims, shape, kind, monkeypatch):
    """Sums that binary64 holds exactly come out exact, zeros included: unit links, and one
    component at one site or small whole numbers everywhere."""
    monkeypatch.setenv("WL_HOP_BLOCK", str(shape))
    psi = torch.zeros_like(fields.gaussian_fermion(dims, 1, 1))
    if kind == "point":
        psi[0, 5, 1, 2] = 1.0
    else:
        psi = torch.view_as_complex(torch.randint(-8, 9, psi.shape + (2,), generator=fields.generator(3)).double())
    for dagger, got, want in _cases(dims, "unit", psi):
        re, im = want.error(got)
        assert not re.any() and not im.any(), dagger


def test_links_round_to_nearest():
    """Small off-diagonal entries of x links come out as the nearest multiples of 2^-59 (ties to even):
    a constant source of colour 1 reaches colour 0 through them alone, and components that small
    next to colour 1 are computed from the links as held."""
    dims = (4, 4, 4, 4)
    V = fields.volume(dims)
    psi = torch.zeros_like(fields.gaussian_fermion(dims, 1, 1))
    psi[..., 0, 1] = 1.0
    gen = np.random.default_rng(5)
    many = gen.uniform(2.0 ** -13, 2.0 ** -6, V) * gen.choice([-1.0, 1.0], V)
    ties = (gen.integers(2 ** 47, 2 ** 51, V) + 0.5) * 2.0 ** -59 * gen.choice([-1.0, 1.0], V)
    few = [k * 2.0 ** -60 for k in (1, 1 + 2.0 ** -52, 1.5, 2, 3, 5, -1, -3, 2.0 ** -3)] + [5e-324, 1e-300]
    for values in [many, ties, np.concatenate([many[:V - 1], [0.0]])] + [np.array([0.0] * 7 + [v] + [0.0] * (V - 8)) for v in few]:
        U = fields.gauge_field(dims, "unit", 0)
        U[:, 0, 0, 1] = torch.from_numpy(values).to(U.dtype)
        with wilson.Gauge(dims, 0.12, U.cuda(), precs=("f64",), bc=BC) as g:
            got = _apply(g, psi.cuda(), 0)[:, 0, 0]
        assert np.array_equal(got.real, np.rint(values * 2.0 ** 59) * 2.0 ** -59) and not got.imag.any()


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("kind", ["all 2^-27", "all 2^-40", "all 2^-66", "one link", "a row", "a column", "zeros"])
def test_small_links(dims, kind):
    """Links, or rows or columns of them, far below 1 keep all their digits.  Plain FP64 passes each
    product through at most 16 roundings (projection 1, product sum 6, hop sum 8): 16 * 2^-53 of
    the sum of the products' moduli (17: second order).  Links that are zero are as good as any."""
    U = fields.gauge_field(dims, "haar", 13)
    psi = fields.gaussian_fermion(dims, 1, 11)
    if kind == "one link":  # and one source, whose only way to site 3 is that link (Ly > 2)
        U[3, 1] *= 2.0 ** -40
        psi[:, [s for s in range(psi.shape[1]) if s != 3 + dims[0]]] = 0.0
    elif kind in ("a row", "a column"):  # of all z links; the sources in one slice, forward of some sites and behind others (Lz > 2)
        U[:, [0, 1, 3]] = 0.0
        U[(slice(None), 2) + ((1, slice(None)) if kind == "a row" else (slice(None), 1))] *= 2.0 ** -40
        psi.reshape(dims[::-1] + (4, 3))[:, [z for z in range(dims[2]) if z != 1]] = 0.0
    elif kind == "zeros":
        U[3, 1], U[4, 2, 1], U[5, 0, :, 2] = 0.0, 0.0, 0.0
    else:
        U *= 2.0 ** int(kind.split("^")[1])
    for dagger, got, want in _cases(dims, U, psi):
        re, im = want.error(got)
        bound = 17 * 2.0 ** -53 * want.total
        assert np.all(np.abs(re) <= bound) and np.all(np.abs(im) <= bound), dagger


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("links", ["haar", "smooth"])
def test_error_of_a_field(dims, shape, links, monkeypatch):
    """Gaussian fields: every component within the steps' bound, and the root mean square of the errors
    no larger than that of the plain FP64 kernels (the links doubled, result halved: exact).

    Bound per component, in units of 2^-53 m, m the largest real component of the site's projected
    neighbours (the scale q is at most 2 m): the sum's 15.5 q are 31, projecting rounds eight times six
    products of a row of norm 1 by 2^-53 m (8 sqrt(6) < 20), and the sum, below 8 sqrt(6) m, is
    rounded once more (20): 71."""
    monkeypatch.setenv("WL_HOP_BLOCK", str(shape))
    psi = fields.gaussian_fermion(dims, 1, 11)
    U = fields.gauge_field(dims, links, 13)
    squares = np.zeros(2)
    for (dagger, got, want), (_, double, _) in zip(_cases(dims, U, psi), _cases(dims, 2 * U, psi)):
        bound = 71 * 2.0 ** -53 * want.largest[:, None, None]
        for k, x in enumerate((got, double / 2)):
            re, im = want.error(x)
            squares[k] += (re ** 2).sum() + (im ** 2).sum()
            assert k or (np.all(np.abs(re) <= bound) and np.all(np.abs(im) <= bound)), dagger
    assert squares[0] <= squares[1], np.sqrt(squares)


@pytest.mark.parametrize("dims", DIMS[:2])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_six_threads_per_site_on_a_partial_tile(dims, nrhs, monkeypatch):
    """D, M_ee and their daggers on 8 and 24 sites a parity, bit for bit those of one thread per site;
    FP64 solves (the reducing forms) to the oracle's residual."""
    kappa = 0.12
    U = fields.gauge_field(dims, "haar", 13)
    psi = fields.gaussian_fermion(dims, nrhs, 11).cuda()
    outs = {}
    for shape in SHAPES:
        monkeypatch.setenv("WL_HOP_BLOCK", str(shape))
        with wilson.Gauge(dims, kappa, U.cuda(), precs=("f64",), bc=BC) as g:
            fb = wilson.wl_field_bytes(g.handle, wilson.WL_F64, 1)
            full = torch.empty(2 * nrhs * fb, dtype=torch.uint8, device="cuda")
            for k in range(2 * nrhs):
                wilson.wl_field_to_internal(g.handle, full[k * fb:(k + 1) * fb], psi[k // 2:k // 2 + 1], k % 2, wilson.WL_F64, 1)
            even = g.field("f64", nrhs)
            wilson.wl_field_to_internal(g.handle, even, psi, 0, wilson.WL_F64, nrhs)
            for eo, x in ((0, full), (1, even)):
                for dagger in (0, 1):
                    out = torch.zeros_like(x)
                    wilson.wilson_mult(g.handle, out, x, eo, dagger, wilson.WL_F64, nrhs)
                    outs.setdefault((eo, dagger), []).append(out.cpu())
            for eo in (False, True):
                x = torch.zeros_like(psi)
                wilson.wilson_solve(g.handle, x, psi, nrhs, wilson.solve_params(tol=1e-10, eo=eo, inner=wilson.WL_F64))
                for r in range(nrhs):
                    tr = oracle.true_residual(U.numpy(), psi[r].cpu().numpy(), x[r].cpu().numpy(), dims, BC, kappa)
                    assert tr <= 1e-10, (shape, eo, r)
    for key, (one, six) in outs.items():
        assert torch.equal(one, six), key


SMALL = ["colours 1e-6", "colours 1e-10", "colours 1e-20", "spins 1e-9", "imaginary 1e-8", "sites", "components"]


def _uneven(dims, kind):
    """A Gaussian field with parts of it scaled down, or scales all over."""
    psi, gen = fields.gaussian_fermion(dims, 1, 11), fields.generator(12)
    if kind.startswith("colours"):
        psi[..., 1:] *= float(kind.split()[1])
    elif kind.startswith("spins"):
        psi[:, :, 1:] *= float(kind.split()[1])
    elif kind.startswith("imaginary"):
        psi = torch.complex(psi.real, psi.imag * float(kind.split()[1]))
    else:
        n = psi.shape[:2] + ((1, 1) if kind == "sites" else (4, 3))
        psi *= 10.0 ** (24 * torch.rand(n, generator=gen, dtype=torch.float64) - 12)
    return psi


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("links", ["unit", "smooth", "haar"])
@pytest.mark.parametrize("kind", SMALL)
def test_small_components(dims, shape, links, kind, monkeypatch):
    """Every component is as accurate as its own terms, also next to larger ones.

    In units of 2^-53 q, q the site's scale, the fixed-point sum is within 15.5 of exact, and a
    component that keeps it has a contribution of at least q / 16, so within 16 * 15.5 = 248 of its
    total; projecting (1) and the final rounding (1) add 2, which leaves 250 < 256 = 2^-45 2^53.
    Components in binary64 pass 16 roundings."""
    monkeypatch.setenv("WL_HOP_BLOCK", str(shape))
    for dagger, got, want in _cases(dims, links, _uneven(dims, kind)):
        re, im = want.error(got)
        bound = 2.0 ** -45 * want.total
        assert np.all(np.abs(re) <= bound) and np.all(np.abs(im) <= bound), dagger


@pytest.mark.parametrize("kind", ["colours 1e-10", "components"])
def test_small_components_of_blocks(kind):
    """The decomposed lattice takes the undivided one's steps, at the cut faces too."""
    dims = (4, 4, 4, 8)
    psi = _uneven(dims, kind).cuda()
    U = fields.gauge_field(dims, "unit", 0).cuda()
    with wilson.Gauge(dims, 0.12, U, precs=("f64",), bc=BC) as g, \
            wilson.Decomposition(dims, 0.12, U, (1, 1, 2, 2), precs=("f64",), bc=BC) as dd:
        want = _apply(g, psi, 0)
        got = _apply_blocks(dd, psi)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("blocks", [1, 2])
def test_links_near_one(blocks):
    """Links 1 + O(1e-8): the way from one colour to another is worth 1e-8, and keeps its digits
    (test_small_components' bound), on the whole lattice and on blocks."""
    dims = (4, 4, 4, 8)
    U = fields.gauge_field(dims, "smooth", 13, eps=1e-8)
    psi = fields.gaussian_fermion(dims, 1, 11)
    psi[..., 1:] = 0.0
    if blocks == 1:
        with wilson.Gauge(dims, 0.12, U.cuda(), precs=("f64",), bc=BC) as g:
            got = _apply(g, psi.cuda(), 0)
    else:
        with wilson.Decomposition(dims, 0.12, U.cuda(), (1, 1, 1, blocks), precs=("f64",), bc=BC) as dd:
            got = _apply_blocks(dd, psi.cuda())
    want = Exact(U.numpy(), psi[0].numpy(), dims, 0)
    re, im = want.error(got)
    bound = 2.0 ** -45 * want.total
    assert np.all(np.abs(re) <= bound) and np.all(np.abs(im) <= bound)


def test_one_colour_in_a_batch():
    """Batched FP64 solves on unit links (links in shared memory): a source of one colour leaves the
    other colours exactly zero, and the true residual is the oracle's."""
    dims, kappa = (4, 4, 4, 6), 0.12
    U = fields.gauge_field(dims, "unit", 0)
    b = fields.gaussian_fermion(dims, 2, 5)
    b[..., 1:] = 0.0
    x = torch.zeros_like(b).cuda()
    with wilson.Gauge(dims, kappa, U.cuda(), precs=("f64",), bc=BC) as g:
        wilson.wilson_solve_batch([g.handle], [x], [b.cuda()], [2], wilson.solve_params(tol=1e-10, inner=wilson.WL_F64))
    x = x.cpu()
    assert not torch.any(x[..., 1:]) and torch.any(x[..., 0])
    for r in range(2):
        assert oracle.true_residual(U.numpy(), b[r].numpy(), x[r].numpy(), dims, BC, kappa) <= 1e-10
