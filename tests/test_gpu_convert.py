"""Layout conversion at the edges of its blocks (64 half sites), for canonical fields
aligned to 16 and to 8 bytes, and the FP64 -> FP32 rounding against IEEE 754's."""
import numpy as np
import pytest
import torch

from paper_1811_00893_gb300 import fields, wilson

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)


def _shifted(shape, shift):
    """A zeroed complex128 tensor whose data starts `shift` doubles into a buffer."""
    n = int(np.prod(shape)) * 2
    return torch.zeros(n + 2, dtype=torch.float64, device="cuda")[shift:shift + n]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 4), (6, 2, 4, 10), (8, 6, 4, 10)])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "df64"])
@pytest.mark.parametrize("shift", [0, 1])
def test_round_trip(dims, prec, shift):
    p, nrhs, V = wilson.PREC[prec], 3, fields.volume(dims)
    U = fields.gauge_field(dims, "unit", 0).cuda()
    psi = fields.gaussian_fermion(dims, nrhs, 5).cuda()
    src, back = _shifted(psi.shape, shift), _shifted(psi.shape, shift)
    src.copy_(torch.view_as_real(psi).reshape(-1))
    with wilson.Gauge(dims, 0.12, U, bc=BC) as g:
        for parity in (0, 1):
            f = g.field(p, nrhs)
            wilson.wl_field_to_internal(g.handle, f, src, parity, p, nrhs)
            wilson.wl_field_to_canonical(g.handle, back, f, parity, p, nrhs)
            if prec == "f32":  # plane k, site i: components 2k, 2k + 1 of the parity's i-th site
                c = fields.site_coords(dims)
                mine = np.flatnonzero(c.sum(1) % 2 == parity)
                want = psi.cpu().numpy().reshape(nrhs, V, 12)[:, mine].reshape(nrhs, -1, 6, 2).transpose(0, 2, 1, 3)
                got = f.view(torch.float32).cpu().numpy().reshape(nrhs, 6, -1, 2, 2)
                assert np.array_equal(got[..., 0], want.real.astype(np.float32)) and np.array_equal(got[..., 1], want.imag.astype(np.float32))
    a, b = src.cpu().numpy(), back.cpu().numpy()
    if prec == "f64":
        assert np.array_equal(a, b)
    elif prec == "f32":
        assert np.array_equal(a.astype(np.float32).astype(np.float64), b)
    else:  # 2^-11 of the site's largest component (binary16, or int16), 2^-47 (double-float)
        m = np.abs(a.reshape(-1, 24)).max(1, keepdims=True)
        assert np.all(np.abs(a - b).reshape(-1, 24) <= m * (2.0 ** -11 if prec == "f16" else 2.0 ** -47))


def test_fp32_rounding():
    """Ties both ways, carries, the ends of the integer-arithmetic range, subnormals, overflow, zeros, non-finite."""
    one = np.float64(1.0)
    ulp = 2.0 ** -23
    v = [one + k * ulp / 4 for k in range(16)] + [2.0 - ulp / 4, 2.0 - ulp / 2, 2.0 - 3 * ulp / 4, 2.0 - 2.0 ** -52]
    v += [s * w for s in (2.0 ** -74, 2.0 ** -75, 2.0 ** -126, 2.0 ** -127, 2.0 ** -149, 2.0 ** -150, 2.0 ** 126, 2.0 ** 127) for w in (1.0, 1.0 + ulp / 2, 2.0 - ulp / 2)]
    v += [0.0, 1e-300, 1e300, np.inf, np.nan, 5e-324, 3.4028235677973366e38]
    v = np.array(v + [-x for x in v], np.float64)
    dims = (4, 4, 4, 4)
    V = fields.volume(dims)
    full = np.resize(v, V * 24)
    with np.errstate(over="ignore", invalid="ignore"):
        want = full.astype(np.float32).astype(np.float64)
    src = torch.from_numpy(full).cuda()
    back = torch.zeros_like(src)
    with wilson.Gauge(dims, 0.12, fields.gauge_field(dims, "unit", 0).cuda(), precs=("f64", "f32"), bc=BC) as g:
        for parity in (0, 1):
            f = g.field("f32")
            wilson.wl_field_to_internal(g.handle, f, src, parity, wilson.WL_F32, 1)
            wilson.wl_field_to_canonical(g.handle, back, f, parity, wilson.WL_F32, 1)
    got = back.cpu().numpy()
    assert np.array_equal(got, want, equal_nan=True) and np.array_equal(np.signbit(got), np.signbit(want) | (np.isnan(want) & np.signbit(got)))
