"""GPU kernels at the edges of their tiles, grids and right-hand-side counts, against the oracle."""
import numpy as np
import pytest

import synthetic as S
from oracle import c_oracle as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F32, F64, Context  # noqa: E402


# grids of one block and of many, blocks of one warp, of a partial last warp and of more
# warps than one combining round, one to twelve columns: a sum that misses or repeats a
# partial sum ends in a residual report that is wrong by far more than rounding
@pytest.mark.parametrize("dims,nrhs,block,tile", [((4, 2, 2, 2), 1, 32, 1), ((4, 4, 4, 6), 1, 256, 1),
                                                  ((8, 6, 4, 10), 5, 64, 1), ((4, 4, 4, 6), 7, 160, 1),
                                                  ((6, 4, 6, 4), 12, 96, 4), ((16, 8, 8, 8), 11, 128, 1),
                                                  ((8, 8, 8, 8), 2, 64, 2)])
@pytest.mark.parametrize("method", ["cg", "bicgstab"])
def test_grid_reductions(dims, nrhs, block, tile, method):
    kappa = 0.11
    U = S.gauge_field(dims, 0.3, 21)
    b = np.stack([S.gaussian_spinor(dims, 60 + r) for r in range(nrhs)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        ctx.gauge_upload(U, 18, F32)
        ctx.set_launch(F32, nrhs, block=block, rhs_tile=tile)
        bd = ctx.to_device(b if nrhs > 1 else b[0], F64, nrhs)
        x = ctx.empty_full(F64, nrhs)
        solve = ctx.cg_solve_multi if method == "cg" else ctx.bicgstab_solve_multi
        infos = solve(x, bd, kappa, nrhs, tol=1e-10, inner_prec=F32)
        xs = ctx.to_host(x, F64, nrhs).reshape((nrhs,) + b.shape[1:])
    for r in range(nrhs):
        res = float(np.linalg.norm(b[r] - C.wilson(U, xs[r], kappa)) / np.linalg.norm(b[r]))
        assert res <= 1e-10
        # both residuals are FP64 sums over the same x: they differ by the rounding of M x,
        # of order 1e-16 of |b|
        assert abs(infos[r].true_rel_residual - res) < 1e-13
