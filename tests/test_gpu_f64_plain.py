"""The FP64 kernels with plain FP64 links.

SU(3) links are held as fixed point, so the other FP64 tests run those kernels.  Here every
gauge object has its links times 1.5, whose largest entries are too large for fixed point, and
kappa over 1.5: the same operator from plain FP64 links.  The tests themselves are those
of the parity, clover, solve, batch and decomposition files, run on such cases in FP64, and
where the outer residuals are in df64 for such links, in the mixed precisions too.
"""
import pytest
import torch

import gpu_helpers
import test_gpu_batch as batch
import test_gpu_clover as clover
import test_gpu_dd as decomposed
import test_gpu_parity as parity
import test_gpu_solve as solves
from paper_1811_00893_gb300 import fields, wilson

pytestmark = pytest.mark.gpu

SCALE = 1.5


class Case(gpu_helpers.Case):
    def __init__(self, dims, kappa=0.12, kind="haar", seed=1, bc=(1, 1, 1, -1), precs=("f64", "f32", "f16")):
        self.dims, self.kappa, self.bc = tuple(dims), kappa / SCALE, bc
        U = SCALE * fields.gauge_field(dims, kind, seed)
        self.U, self.U_dev = U.numpy(), U.cuda().contiguous()
        self.g = wilson.Gauge(dims, self.kappa, self.U_dev, precs=precs, bc=bc)
        self.V = self.U.shape[0]
        self.Vh = self.V // 2


class DDCase(decomposed.DDCase):
    def __init__(self, dims, grid, bc, kappa=0.124, seed=3):
        self.dims, self.grid, self.bc, self.kappa = tuple(dims), tuple(grid), bc, kappa / SCALE
        U = SCALE * fields.gauge_field(dims, "haar", seed)
        self.U, self.U_dev = U.numpy(), U.cuda().contiguous()
        self.dd = wilson.Decomposition(dims, self.kappa, self.U_dev, grid, precs=("f64", "f32"), bc=bc)
        self.V = self.U.shape[0]


@pytest.fixture
def plain(monkeypatch):
    """The tests of the parity and batch files make their cases by this name."""
    monkeypatch.setattr(parity, "Case", Case)
    monkeypatch.setattr(batch, "Case", Case)
    return monkeypatch


@pytest.fixture(scope="module", params=parity.SMALL, ids=lambda c: "x".join(map(str, c[0])))
def case(request):
    dims, bc = request.param
    c = Case(dims, kappa=0.124, seed=7, bc=bc)
    yield c
    c.close()


def test_link_form(monkeypatch, capfd):
    """Autotuned launches name their link form: 0 here, 3 for the same links unscaled."""
    monkeypatch.setenv("WL_AUTOTUNE_VERBOSE", "1")
    for kind, form in ((Case, "l0"), (gpu_helpers.Case, "l3")):
        c = kind((4, 4, 4, 4))
        capfd.readouterr()
        out = c.g.field("f64")
        wilson.wilson_dslash(c.g.handle, out, c.to_internal(c.source(), 1, "f64"), 0, 0, wilson.WL_F64, 1)
        lines = [s for s in capfd.readouterr().err.splitlines() if "hop p0" in s]
        assert len(lines) == 1 and form in lines[0].split(), lines
        c.close()


@pytest.mark.parametrize("dagger", [0, 1])
def test_operators(case, dagger):
    parity.test_dslash_matches_oracle(case, "f64", dagger)
    parity.test_full_D_matches_oracle(case, "f64", dagger)
    parity.test_Mee_matches_oracle(case, "f64", dagger)


@pytest.mark.parametrize("shape", [1, 2, 3, 3064, 3128, 3256])
def test_multi_rhs_shapes(plain, shape):
    parity.test_wide_multi_rhs_shapes_match_oracle(plain, "f64", shape)


def test_rhs_beyond_one_launch_chunk(plain):
    parity.test_rhs_beyond_one_launch_chunk("f64")


@pytest.mark.parametrize("shape", [32, 64, 256, 1032, 1064, 1128])
def test_reducing_shapes(plain, shape):
    parity.test_reducing_hop_shapes_in_solve(plain, shape)


@pytest.mark.parametrize("dims", [(6, 4, 2, 6), (6, 4, 4, 6), (4, 4, 4, 4)])
def test_three_threads_per_site(plain, dims):
    """hop_rows_kernel against one thread per site, bit for bit, and against the oracle."""
    parity.test_fp64_rows_kernel_equals_one_thread_per_site(plain, dims)


def test_three_threads_per_site_in_solves(plain):
    parity.test_fp64_rows_kernel_in_solves(plain)


@pytest.mark.parametrize("dims,bc", clover.SMALL[:2], ids=["4x4x4x4", "6x4x2x8"])
def test_clover(dims, bc):
    c = Case(dims, kappa=0.124, seed=7, bc=bc)
    try:
        c.F_dev = fields.clover_field(dims, 57).cuda().contiguous()
        c.F = c.F_dev.cpu().numpy()
        wilson.wl_clover_set(c.g.handle, c.F_dev)
        for dagger in (0, 1):
            clover.test_clover_D_matches_oracle(c, "f64", dagger)
            clover.test_clover_Mee_matches_oracle(c, "f64", dagger)
        for eo, inner in ((False, wilson.WL_F64), (True, wilson.WL_F64), (True, wilson.WL_F32)):
            clover.test_clover_solve_reaches_true_residual(c, eo, inner, 0.0)
    finally:
        c.close()


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("scheme", sorted(solves.SCHEMES))
def test_solves(scheme, nrhs):
    c = Case((6, 4, 4, 8), seed=1000)
    try:
        b = c.source(nrhs=nrhs, seed=2000)
        x = torch.zeros_like(b)
        rc, infos = wilson.wilson_solve(c.g.handle, x, b, nrhs, wilson.solve_params(tol=1e-10, **solves.SCHEMES[scheme]))
        solves.check_solution(c, b, x, infos)
    finally:
        c.close()


@pytest.mark.parametrize("inner,delta,graph", [(wilson.WL_F32, 0.0, 0), (wilson.WL_F16, 0.1, 0), (wilson.WL_F64, 0.0, 2)],
                         ids=["f32", "f16-reliable", "f64-graph"])
def test_batch(plain, inner, delta, graph):
    batch.test_small_uneven_batch(inner, delta, graph)


def test_batch_of_both_forms(monkeypatch):
    """Lattices with fixed-point and with plain links in one FP64 batch."""
    kinds = iter([gpu_helpers.Case, Case, gpu_helpers.Case, Case])
    monkeypatch.setattr(batch, "Case", lambda *a, **k: next(kinds)(*a, **k))
    batch.test_small_uneven_batch(wilson.WL_F64, 0.0, 2)


@pytest.mark.parametrize("dims,grid,bc", decomposed.CASES[1:4], ids=["t", "tz", "tzy"])
def test_blocks(dims, grid, bc):
    c = DDCase(dims, grid, bc)
    try:
        for dagger in (0, 1):
            decomposed.test_dslash_dd_matches_oracle(c, "f64", dagger)
            decomposed.test_mult_dd_matches_oracle(c, "f64", dagger)
        decomposed.test_dslash_dd_equals_undivided(c, "f64")
        for inner in ("f64", "f32"):
            decomposed.test_solve_dd_reaches_oracle_residual(c, inner, 0.0)
    finally:
        c.close()
