"""Batches whose lattice lookup takes two loads per lane (more than 32 lattices) and whose
activity lookup takes a whole warp (32 right-hand sides), tiles partly filled: every system
reaches a true residual of 1e-10 under the oracle's FP64 D."""
import pytest
import torch

from paper_1811_00893_gb300 import wilson
from test_gpu_batch import TOL, check, make_batch

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2, 2), (4, 4, 4, 4), (4, 2, 2, 6)]


@pytest.mark.parametrize("nlat", [1, 32, 33, 64])
@pytest.mark.parametrize("inner,delta", [(wilson.WL_F32, 0.0), (wilson.WL_F16, 0.1)], ids=["f32", "f16"])
def test_many_lattices(nlat, inner, delta):
    specs = [(DIMS[n % 3], 32 if n == nlat - 1 else 1 + n % 2, 0.11 + 0.0002 * n) for n in range(nlat)]
    cases, bs = make_batch(specs)
    try:
        xs = [torch.zeros_like(b) for b in bs]
        p = wilson.solve_params(tol=TOL, eo=True, inner=inner, delta=delta)
        rc, infos = wilson.wilson_solve_batch([c.g.handle for c in cases], xs, bs, [b.shape[0] for b in bs], p)
        assert rc == 0
        check(cases, bs, xs, infos)
    finally:
        for c in cases:
            c.close()
