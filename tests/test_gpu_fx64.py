"""FP64 hopping term with fixed-point links against the plain FP64 kernels.

Links whose entries exceed a modulus of 1.25 keep plain FP64 arithmetic, and the hopping
term is linear in the links, so a gauge object with the links doubled (an exact scaling)
gives the FP64 kernels' result for the same input.  Both sides are compared site by site.

Tolerance per site, against m, the largest |real component| of its eight neighbours: a
projected component is at most 2 m, and a component of the site sum adds 8 x 3 complex
products of a link row (norm 1) with a projected colour vector (norm <= 2 sqrt(6) m), so
sum |W| |h| <= 8 * 2 sqrt(6) m < 40 m.  FP64 passes each term through at most 16 roundings
(projection 1, product sum 6, hop sum 8, the doubling none): 16 * 2^-53 * 40 m = 640 * 2^-53 m.
The fixed-point sum stays below 16 units of 2^-53 m.  2^-43 m covers both.
"""
import numpy as np
import pytest
import torch

from paper_1811_00893_gb300 import fields, wilson

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -43
BC = (1, 1, 1, -1)


def _pick(cond, a, b):
    return torch.where(cond, torch.tensor(a, dtype=torch.float64), torch.tensor(b, dtype=torch.float64))


def _source(kind, dims):
    V = fields.volume(dims)
    psi = fields.gaussian_fermion(dims, 1, 11)
    gen = fields.generator(12)
    if kind == "zero":
        psi.zero_()
    elif kind == "point":
        keep = psi[0, 5].clone()
        psi.zero_()
        psi[0, 5] = keep
    elif kind == "tiny":  # above and below the fixed-point range (2^-953 ~ 1e-287)
        psi *= _pick(torch.rand(V, generator=gen, dtype=torch.float64) < 0.5, 1e-280, 1e-295)[None, :, None, None]
    elif kind == "subnormal":
        psi *= 1e-310
    elif kind == "huge":  # some sites above 2^1007 ~ 1e303
        psi *= _pick(torch.rand(V, generator=gen, dtype=torch.float64) < 0.9, 1.0, 1e304)[None, :, None, None]
    elif kind == "mixed":  # neighbours of very different scales
        psi *= 10.0 ** (60 * torch.rand(V, generator=gen, dtype=torch.float64) - 30)[None, :, None, None]
    elif kind == "spread":  # components of very different scales
        psi = torch.view_as_complex(torch.view_as_real(psi) * 10.0 ** (30 * torch.rand(1, V, 4, 3, 2, generator=gen, dtype=torch.float64) - 15))
    elif kind == "inf":
        psi[0, 7, 1, 2] = complex(float("inf"), 1.0)
    elif kind == "nan":
        psi[0, 7, 1, 2] = complex(float("nan"), 1.0)
    return psi


def _apply(g, psi, dagger):
    """The hopping term on both parities: (V, 24) reals of the canonical field."""
    out = torch.zeros_like(psi)
    for p in (0, 1):
        i, o = g.field("f64"), g.field("f64")
        wilson.wl_field_to_internal(g.handle, i, psi, 1 - p, wilson.WL_F64, 1)
        wilson.wilson_dslash(g.handle, o, i, p, dagger, wilson.WL_F64, 1)
        wilson.wl_field_to_canonical(g.handle, out, o, p, wilson.WL_F64, 1)
    return torch.view_as_real(out)[0].cpu().numpy().reshape(-1, 24)


def _neighbour_max(psi, dims):
    """max |real component| over each site's eight neighbours."""
    m = np.abs(np.ascontiguousarray(psi.cpu().numpy()[0]).view(np.float64).reshape(-1, 24)).max(1)
    m = np.where(np.isfinite(m), m, np.inf).reshape(dims[::-1])
    return np.maximum.reduce([np.roll(m, s, ax) for ax in range(4) for s in (1, -1)]).reshape(-1)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 2, 4, 10)])
@pytest.mark.parametrize("kind", ["gauss", "zero", "point", "tiny", "subnormal", "huge", "mixed", "spread", "inf", "nan"])
@pytest.mark.parametrize("shape", [64, 2000])
def test_against_fp64_kernels(dims, kind, shape, monkeypatch):
    monkeypatch.setenv("WL_HOP_BLOCK", str(shape))
    psi = _source(kind, dims).cuda()
    U = fields.gauge_field(dims, "haar", 13).cuda()
    m = _neighbour_max(psi, dims)
    for dagger in (0, 1):
        with wilson.Gauge(dims, 0.12, U, precs=("f64",), bc=BC) as g, wilson.Gauge(dims, 0.12, 2 * U, precs=("f64",), bc=BC) as g2:
            got, want = _apply(g, psi, dagger), _apply(g2, psi, dagger)
        with np.errstate(over="ignore", invalid="ignore"):
            got = 2 * got
            same = np.isfinite(want)
            assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
            # (2^-1070: subnormal results round to multiples of 2^-1074, eight hops on each side)
            bound = (TOL * m + 2.0 ** -1070)[:, None]
            assert np.all(np.abs(got - want)[same] <= np.broadcast_to(bound, same.shape)[same])
        if kind in ("inf", "nan"):
            assert not same.all() and same.any()


@pytest.mark.parametrize("scale", [1.25, 0.0078125])
def test_link_scale(scale):
    """Entries up to the largest modulus that fits, and small ones."""
    dims = (4, 4, 4, 6)
    U = fields.gauge_field(dims, "unit", 0).cuda()
    psi = _source("gauss", dims).cuda()
    with wilson.Gauge(dims, 0.12, scale * U, precs=("f64",), bc=BC) as g, wilson.Gauge(dims, 0.12, 2 * U, precs=("f64",), bc=BC) as g2:
        got, want = _apply(g, psi, 0), _apply(g2, psi, 0) * (scale / 2)
    assert np.all(np.abs(got - want) <= scale * (TOL * _neighbour_max(psi, dims))[:, None])


def test_one_block_does_not_fit():
    """A link too large for fixed point in one block: every block takes plain FP64 arithmetic."""
    dims = (4, 4, 4, 8)
    U = fields.gauge_field(dims, "haar", 13).cuda()
    U[3] *= 4.0
    psi = _source("gauss", dims).cuda()
    with wilson.Gauge(dims, 0.12, U, precs=("f64",), bc=BC) as g, \
            wilson.Decomposition(dims, 0.12, U, (1, 1, 1, 2), precs=("f64",), bc=BC) as dd:
        want = _apply(g, psi, 0)
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
    assert np.array_equal(torch.view_as_real(got)[0].cpu().numpy().reshape(-1, 24), want)
