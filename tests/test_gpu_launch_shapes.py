"""Hand-set launches of the operator at the limits of a block's shared memory, in every
launch a solve makes with them."""
import numpy as np
import pytest

import synthetic as S
from gpuhelp import TOL, gpu_hopping_full, rel
from oracle import c_oracle as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F16, F32, F64, Context, PLQError  # noqa: E402
from paper_1405_0700_gb300 import plq  # noqa: E402

KAPPA = 0.115


def solve_and_check(ctx, U, b, method="cg"):
    n = len(b)
    x = ctx.empty_full(F64, n)
    fn = ctx.cg_solve_multi if method == "cg" else ctx.bicgstab_solve_multi
    fn(x, ctx.to_device(b, F64, n), KAPPA, n, inner_prec=F32)
    xs = ctx.to_host(x, F64, n).reshape(b.shape)
    for r in range(n):
        assert np.linalg.norm(b[r] - C.wilson(U, xs[r], KAPPA)) <= 1e-10 * np.linalg.norm(b[r])


# links and copied neighbour spinors of a block take 45-47 KB: below 48 KB alone, above with
# the shared memory of a reduction (3 RHS x 32 sites, 12 x 16, 8 x 16)
@pytest.mark.parametrize("nrhs,block,smem", [(3, 96, 3), (12, 192, 2), (12, 256, 2), (8, 128, 3), (7, 128, 3)])
@pytest.mark.parametrize("reals", [18, 12])
def test_solve_with_a_block_near_48_kb(nrhs, block, smem, reals):
    dims = (8, 4, 4, 4)
    U = S.gauge_field(dims, 0.3, 61)
    b = np.stack([S.gaussian_spinor(dims, 62 + r) for r in range(nrhs)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        ctx.gauge_upload(U, reals, F32)
        ctx.set_launch(F32, nrhs, block, smem_links=smem)
        solve_and_check(ctx, U, b)


def test_large_block_after_a_smaller_one():
    """130 KB, 80 KB, 130 KB again, in the plain and in the reducing launches."""
    dims = (4, 4, 4, 6)
    U = S.gauge_field(dims, 0.3, 63)
    b = np.stack([S.gaussian_spinor(dims, 64 + r) for r in range(12)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        ctx.gauge_upload(U, 18, F32)
        for block in (1024, 192, 1024):
            ctx.set_launch(F32, 12, block, smem_links=3)
            H = gpu_hopping_full(ctx, b, F32, 12).reshape(b.shape)
            for r in range(12):
                assert rel(H[r], C.hopping(U, b[r])) <= TOL[F32]
            solve_and_check(ctx, U, b)


# rows of which 8 (300 elements) or 5 (480) fill all but 2048 bytes of a block's shared memory,
# less than the norm epilogue needs for itself
@pytest.mark.parametrize("lx,reals", [(50, 18), (80, 12)])
def test_row_streamed_solve_with_full_shared_memory(lx, reals):
    dims = (4, lx, 2, 2)
    U = S.gauge_field(dims, 0.3, 65)
    b = np.stack([S.gaussian_spinor(dims, 66 + r) for r in range(12)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        ctx.gauge_upload(U, reals, F32)
        ctx.set_launch(F32, 12, smem_links=4)
        solve_and_check(ctx, U, b)
        for slots in (2, 3):  # slots, not sites per thread of the launches that kernel does not make
            ctx.set_launch(F32, 12, smem_links=4, sites_per_thread=slots)
            for method in ("cg", "bicgstab"):
                solve_and_check(ctx, U, b, method)


# what plq_autotune may report can be set by hand: the split kernel, in the one form it has
@pytest.mark.parametrize("prec,nrhs", [(F64, 1), (F32, 1), (F16, 1), (F64, 3), (F32, 3), (F32, 12)])
def test_split_launch_by_hand(prec, nrhs):
    dims = (4, 4, 6, 4)
    U = S.gauge_field(dims, 0.3, 67)
    b = np.stack([S.gaussian_spinor(dims, 68 + r) for r in range(nrhs)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        if prec != F64:
            ctx.gauge_upload(U, 18, prec)
        ctx.set_launch(prec, nrhs, 256, smem_links=5)
        H = gpu_hopping_full(ctx, b if nrhs > 1 else b[0], prec, nrhs).reshape(b.shape)
        for r in range(nrhs):
            assert rel(H[r], C.hopping(U, b[r])) <= TOL[prec]
        x = ctx.empty_full(F64, nrhs)
        bd = ctx.to_device(b if nrhs > 1 else b[0], F64, nrhs)
        for solve in (ctx.cg_solve_multi, ctx.bicgstab_solve_multi):  # (its reductions take one right-hand side)
            solve(x, bd, KAPPA, nrhs, inner_prec=prec)
            xs = ctx.to_host(x, F64, nrhs).reshape(b.shape)
            for r in range(nrhs):
                assert np.linalg.norm(b[r] - C.wilson(U, xs[r], KAPPA)) <= 1e-10 * np.linalg.norm(b[r])
        tuned = ctx.autotune(prec, nrhs)
        ctx.set_launch(prec, nrhs, *(tuned[k] for k in ("block", "index_mode", "rhs_tile", "z_chunk", "smem_links",
                                                        "sites_per_thread")))
        for bad in [dict(block=128), dict(index_mode=1), dict(z_chunk=2), dict(sites_per_thread=1), dict(block=0)]:
            with pytest.raises(PLQError) as e:
                ctx.set_launch(prec, nrhs, **dict(dict(block=256, smem_links=5), **bad))
            assert e.value.status == plq.PLQ_ERR_ARG
