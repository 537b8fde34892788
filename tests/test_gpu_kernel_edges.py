"""GPU kernels at the edges of their tiles, grids and right-hand-side counts, against the oracle."""
import numpy as np
import pytest

import synthetic as S
from gpuhelp import TOL, gpu_hopping_full, rel
from oracle import c_oracle as C
from oracle import wilson as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F16, F32, F64, Context, PLQError  # noqa: E402
from paper_1405_0700_gb300 import plq  # noqa: E402


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


# blocks that hold fewer pairs of sites than the lattice leaves them (4x2x2x2: one block;
# 6x10x2x14: ragged last blocks), one to twelve right-hand sides
@pytest.mark.parametrize("dims", [(4, 2, 2, 2), (6, 10, 2, 14), (4, 6, 4, 2)])
@pytest.mark.parametrize("nrhs", [1, 2, 5, 12])
@pytest.mark.parametrize("prec", [F64, F32, F16])
def test_pack_and_unpack(dims, nrhs, prec):
    T, Lx, Ly, Lz = dims
    rng = np.random.default_rng(7)
    phi = rng.standard_normal((nrhs, T, Lz, Ly, Lx, 12, 2)).view(np.complex128)[..., 0]
    t, z, y, x = np.meshgrid(*[np.arange(k) for k in (T, Lz, Ly, Lx)], indexing="ij")
    parity = (t + x + y + z) % 2
    with Context(dims) as ctx:
        full = ctx.to_device(phi if nrhs > 1 else phi[0], prec, nrhs)
        back = ctx.to_host(full, prec, nrhs).reshape(phi.shape[:5] + (12,))
        halves = [h.cpu().numpy() for h in ctx.halves(full, prec, nrhs)]
    Vh = T * Lx * Ly * Lz // 2
    for p in (0, 1):
        ref = phi[:, parity == p].transpose(1, 0, 2)  # (Vh, nrhs, 12): sites in checkerboard order
        if prec == F64:
            got = halves[p].view(np.float64).reshape(12, Vh, nrhs, 2)
            assert np.array_equal(got[..., 0] + 1j * got[..., 1], ref.transpose(2, 0, 1))
        elif prec == F32:
            got = halves[p].view(np.float32).reshape(6, Vh, nrhs, 2, 2).transpose(1, 2, 0, 3, 4).reshape(Vh, nrhs, 12, 2)
            assert np.array_equal(got, ref.astype(np.complex64).view(np.float32).reshape(Vh, nrhs, 12, 2))
        else:
            norms = halves[p][48 * Vh * nrhs:].view(np.float32).reshape(Vh, nrhs)
            r32 = ref.astype(np.complex64).view(np.float32).reshape(Vh, nrhs, 24)
            assert np.array_equal(norms, np.abs(r32).max(axis=2))
    # FP64 exact; FP32 to half an ulp; FP16 to half an ulp of the site's largest component
    tol = {F64: 0.0, F32: 2.0**-24, F16: 2.0**-10}[prec]
    assert np.abs(back - phi).max() <= tol * np.sqrt(2) * np.abs(phi).max()


@pytest.mark.parametrize("what,accepted", [("none", True), ("1e-11 in row 0", False), ("1e-11 in row 2", False),
                                           ("5e-13 in row 2", True), ("1e-11 row 1 phase", False)])
@pytest.mark.parametrize("dims", [(4, 2, 2, 2), (2, 6, 4, 10)])
def test_su3_check_of_twelve_real_links(what, accepted, dims):
    U = S.gauge_field(dims, 0.3, 3)
    u = U[-1, -1, -1, -1, 3]  # the last link of the lattice
    if what == "1e-11 in row 0":
        u[0, 1] += 1e-11
    elif what == "1e-11 in row 2":
        u[2, 2] += 1e-11j
    elif what == "5e-13 in row 2":  # below the limit, above the short test's
        u[2, 0] += 5e-13 * u[2, 1] / abs(u[2, 1])
    elif what == "1e-11 row 1 phase":  # rows stay orthonormal, row 2 no longer their product
        u[1] *= np.exp(1e-11j)
    with Context(dims) as ctx:
        if accepted:
            ctx.gauge_upload(U, 12, F32)
        else:
            with pytest.raises(PLQError) as e:
                ctx.gauge_upload(U, 12, F32)
            assert e.value.status == plq.PLQ_ERR_ARG


# the split kernel (eight warps per 32 elements), the default for FP64 storage and small
# lattices: a last block of fewer elements (16 sites; 5 right-hand sides), the largest FP32
# lattice it takes and the first it does not, and an odd number of sites per block
@pytest.mark.parametrize("dims,nrhs", [((4, 2, 2, 2), 1), ((2, 2, 2, 4), 5), ((6, 10, 2, 6), 1), ((16, 8, 8, 16), 1),
                                       ((16, 10, 8, 14), 1), ((4, 4, 6, 4), 12)])
@pytest.mark.parametrize("prec,reals", [(F64, 18), (F64, 12), (F32, 18), (F32, 12), (F16, 18), (F16, 12)])
def test_split_kernel(dims, nrhs, prec, reals):
    kappa = 0.12
    U = S.gauge_field(dims, 0.3, 31)
    phi = np.stack([S.gaussian_spinor(dims, 80 + r) for r in range(nrhs)])
    with Context(dims) as ctx:
        ctx.gauge_upload(U, reals, prec)
        H = gpu_hopping_full(ctx, phi if nrhs > 1 else phi[0], prec, nrhs).reshape(phi.shape)
        for r in range(nrhs):
            assert rel(H[r], C.hopping(U, phi[r])) <= TOL[prec]
        if nrhs == 1:  # epilogues, both signs of the projectors
            full, out = ctx.to_device(phi[0], prec), ctx.empty_full(prec)
            ctx.twisted_apply(out, full, kappa, 0.3, prec)
            g5 = np.array([1.0, 1, -1, -1])[:, None]
            want = phi[0] - kappa * C.hopping(U, phi[0]) + 2j * kappa * 0.3 * g5 * phi[0]
            assert rel(ctx.to_host(out, prec), want) <= TOL[prec]
            e_in, e_out, tmp = ctx.halves(full, prec)[0], ctx.halves(out, prec)[0], ctx.empty_half(prec)
            t, z, y, x = np.indices(phi.shape[1:5])
            even = ((t + x + y + z) % 2 == 0)[..., None, None]
            for dagger in (False, True):
                ctx.schur_apply(e_out, e_in, tmp, kappa, prec, dagger=dagger)
                v = np.where(even, g5 * phi[0] if dagger else phi[0], 0)
                w = v - kappa**2 * C.hopping(U, C.hopping(U, v))
                got = ctx.to_host(out, prec)[even[..., 0, 0]]
                assert rel(got, (g5 * w if dagger else w)[even[..., 0, 0]]) <= TOL[prec]


def test_calls_follow_the_current_stream():
    """Calls without a stream go to torch's current stream of the current device."""
    side = torch.cuda.Stream()
    assert plq._stream(None) == torch.cuda.current_stream().cuda_stream
    for _ in range(2):
        with torch.cuda.stream(side):
            assert plq._stream(None) == side.cuda_stream == torch.cuda.current_stream().cuda_stream
        assert plq._stream(None) == torch.cuda.current_stream().cuda_stream
    assert plq._stream(side) == side.cuda_stream and plq._stream(5) == 5


# the inner products, search-space slots and restarts of EigCG: one vector, counts around the
# 16 of a launch, restarts every two iterations, fields of less than a block and of several
# elements a thread.  Eigenvalues of H = U^H A U lie within the spectrum of A up to
# |U^H U - 1| <= k 4 2^-24 < 1e-5 (k <= 40 vectors orthonormalised in FP32); a sum that misses
# a term, a slot overwritten or a restart from the wrong slots leaves vectors that are not
# orthonormal or an H that is not theirs.
@pytest.mark.parametrize("dims,unit,nev,m,solves", [((4, 2, 2, 2), False, 1, 4, 18), ((4, 4, 2, 6), False, 6, 14, 6),
                                                    ((16, 8, 8, 16), True, 8, 20, 3)])
def test_eigcg_basis(dims, unit, nev, m, solves):
    kappa = 0.115
    U = S.gauge_field(dims, 0.3, 23)
    if unit:  # free field: A is diagonal in momentum space, 1 - kappa^2 H(p)^2 with H(p) = a +- i |b|
        U = np.zeros_like(U) + np.eye(3)
        # (antiperiodic in time: half-integer momenta)
        p = np.meshgrid(*[2 * np.pi * (np.arange(n) + 0.5 * (i == 0)) / n for i, n in enumerate(dims)], indexing="ij")
        h = 2 * sum(np.cos(q) for q in p) + 2j * np.sqrt(sum(np.sin(q) ** 2 for q in p))
        lam = np.abs(1 - kappa**2 * h**2) ** 2
    else:
        even = W.parity(S.lattice_shape(dims)) == 0
        n = int(even.sum()) * 12
        A = np.empty((n, n), dtype=np.complex128)
        for k in range(n):
            v = np.zeros(S.lattice_shape(dims) + (4, 3), dtype=np.complex128)
            v[even] = np.eye(n)[k].reshape(-1, 4, 3)
            A[:, k] = W.schur_dag(U, W.schur(U, v, kappa), kappa)[even].ravel()
        lam = np.linalg.eigvalsh(A)
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        eig = plq.EigCG(ctx, nev=nev, m=m, max_vectors=nev * solves)
        x = ctx.empty_full(F64)
        for k in range(solves + 1):
            info = eig.solve(x, ctx.to_device(S.gaussian_spinor(dims, 700 + k), F64), kappa, tol=1e-11)
            # |r_x| <= |Mhat^-dag| |r_normal|, |rhs| <= |Mhat| |bhat| and |bhat| <= (1 + 8 kappa) |b|
            assert info.true_rel_residual <= 1.01e-11 * np.sqrt(lam.max() / lam.min()) * (1 + 8 * kappa)
        held, H = eig.vectors, eig.projected_matrix()
        eig.close()
    assert held == nev * solves
    theta = np.linalg.eigvalsh(H)
    assert np.allclose(H, H.conj().T, atol=1e-14)
    assert theta[0] >= lam.min() * (1 - 1e-5) and theta[-1] <= lam.max() * (1 + 1e-5), (theta[0], lam.min())
