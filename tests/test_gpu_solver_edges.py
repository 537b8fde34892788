"""Solver iterations that end early: coefficients that are not finite, iteration caps."""
import numpy as np
import pytest

import synthetic as S
from oracle import c_oracle as C
from oracle import wilson as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F32, F64, Context  # noqa: E402
from paper_1405_0700_gb300 import plq  # noqa: E402

KAPPA = 0.12


def overflowing_system():
    """Two halves of a lattice without links between them, and spatial links of 1e308 (1 + i)
    six time slices from a source of 1e20 on slice 0: CG reaches them in its third
    iteration, whose |Mhat p|^2 is NaN (overflows of either sign are added) while |r|^2 is
    finite.  Returns links, source and the iterate x_e after two iterations."""
    dims = (32, 4, 2, 2)
    U = S.gauge_field(dims, 0.3, 41)
    U[15, ..., 0, :, :] = U[31, ..., 0, :, :] = 0
    U[6, ..., 1:, :, :] = 1e308 * (1 + 1j)
    b = np.zeros(S.lattice_shape(dims) + (4, 3), complex)
    b[0] = 1e20 * S.gaussian_spinor(dims, 42)[0]
    even = (W.parity(S.lattice_shape(dims)) == 0)[..., None, None]
    g5 = np.array([1.0, 1, -1, -1])[:, None]

    def mhat(v):
        return v - KAPPA**2 * np.where(even, C.hopping(U, np.where(even, 0, C.hopping(U, v))), 0)

    def norm2(v):
        return np.sum(v.real**2) + np.sum(v.imag**2)

    bhat = np.where(even, b + KAPPA * C.hopping(U, np.where(even, 0, b)), 0)
    r = g5 * mhat(g5 * bhat)
    x, p, rho = np.zeros_like(r), r, norm2(r)
    with np.errstate(all="ignore"):
        for k in range(3):
            mp = mhat(p)
            alpha = rho / norm2(mp)
            if k == 2:
                assert np.isfinite(rho) and np.isnan(alpha)
                break
            x = x + alpha * p
            r = r - alpha * (g5 * mhat(g5 * mp))
            rho, last = norm2(r), rho
            p = r + rho / last * p
    return dims, U, b, even, x


@pytest.mark.parametrize("solver", ["cg", "cg of two right-hand sides", "eigcg"])
def test_alpha_not_finite_leaves_the_last_iterate(solver):
    dims, U, b, even, want = overflowing_system()
    other = np.zeros_like(b)
    other[16:] = S.gaussian_spinor(dims, 43)[16:]
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        n = 2 if solver.startswith("cg of") else 1
        src = ctx.to_device(np.stack([b, other]) if n == 2 else b, F64, n)
        x = ctx.empty_full(F64, n)
        if solver == "eigcg":
            eig = plq.EigCG(ctx, nev=2, m=12, max_vectors=4)
            info = eig.solve(x, src, KAPPA, tol=1e-8, raise_on_error=False)
            eig.close()
        elif n == 2:
            infos = ctx.cg_solve_multi(x, src, KAPPA, 2, raise_on_error=False)
            info = infos[0]
            assert infos[1].status == plq.PLQ_OK
        else:
            info = ctx.cg_solve(x, src, KAPPA, raise_on_error=False)
        xs = ctx.to_host(x, F64, n).reshape((n,) + b.shape)
    assert info.status == plq.PLQ_ERR_NAN
    e = even[..., 0, 0]
    # two iterations of well-conditioned sums: a few hundred roundings of 2^-53
    assert np.linalg.norm(xs[0][e] - want[e]) <= 1e-13 * np.linalg.norm(want[e])
    if solver != "eigcg":
        assert info.iterations == 2
    if n == 2:
        upper = U.copy()
        upper[6, ..., 1:, :, :] = 0  # (the other half of the lattice does not see these links)
        assert np.linalg.norm(other - C.wilson(upper, xs[1], KAPPA)) <= 1e-10 * np.linalg.norm(other)


# caps around the iterations of one pass of the device loop, and below, at and above what the
# solve needs: the loop's own bound never shows (it would be PLQ_ERR_STATE)
@pytest.mark.parametrize("method,inner,nrhs", [("cg", F64, 1), ("cg", F32, 1), ("cg", F32, 3), ("bicgstab", F32, 1),
                                               ("bicgstab", F64, 2)])
def test_iteration_cap(method, inner, nrhs):
    dims = (8, 4, 4, 4)
    U = S.gauge_field(dims, 0.3, 51)
    b = np.stack([S.gaussian_spinor(dims, 52 + r) for r in range(nrhs)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        if inner != F64:
            ctx.gauge_upload(U, 18, inner)
        src = ctx.to_device(b if nrhs > 1 else b[0], F64, nrhs)
        x = ctx.empty_full(F64, nrhs)

        def solve(maxit):
            fn = ctx.cg_solve_multi if method == "cg" else ctx.bicgstab_solve_multi
            return fn(x, src, KAPPA, nrhs, inner_prec=inner, maxit=maxit, raise_on_error=False)

        need = solve(20000)
        assert all(i.status == plq.PLQ_OK for i in need)
        most = max(i.iterations for i in need)
        for maxit in [1, 2, 3, 4, 5, 6, 7, most - 1, most, most + 1]:
            for i, full in zip(solve(maxit), need):
                assert i.iterations <= maxit
                if maxit >= most:
                    assert i.status == plq.PLQ_OK and i.iterations == full.iterations
                elif maxit <= 7:
                    assert i.status == plq.PLQ_ERR_NOT_CONVERGED and i.iterations == maxit
                else:  # (the residual check behind the last iteration may find it converged)
                    assert i.status in (plq.PLQ_OK, plq.PLQ_ERR_NOT_CONVERGED)
