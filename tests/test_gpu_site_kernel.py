"""The one-thread-per-site operator kernel on small lattices, where the library's own choice is the
split kernel: hand-set launches, every format, epilogue, twist and sign, against the oracle."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import synthetic as S
from gpuhelp import TOL, gpu_hopping_full, rel
from oracle import c_oracle as C
from oracle import wilson as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F16, F32, F64, Context  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
FORMATS = [(F64, 18), (F64, 12), (F32, 18), (F32, 12), (F16, 18), (F16, 12)]


@pytest.mark.parametrize("dims", [(10, 4, 6, 8), (4, 2, 2, 2)])
@pytest.mark.parametrize("prec,reals", FORMATS)
@pytest.mark.parametrize("mode", [0, 1])
def test_operators(dims, prec, reals, mode):
    kappa, mu = 0.12, 0.05
    U, phi = S.gauge_and_spinor(dims, 0.3, 3)
    even = W.parity(S.lattice_shape(dims)) == 0
    half = np.where(even[..., None, None], phi, 0)
    with Context(dims) as ctx:
        ctx.gauge_upload(U, reals, prec)
        ctx.set_launch(prec, 1, 128, index_mode=mode)
        assert rel(gpu_hopping_full(ctx, phi, prec), W.hopping(U, phi)) <= TOL[prec]
        full, out = ctx.to_device(phi, prec), ctx.empty_full(prec)
        ctx.wilson_apply(out, full, kappa, prec)
        assert rel(ctx.to_host(out, prec), W.wilson(U, phi, kappa)) <= TOL[prec]
        ctx.twisted_apply(out, full, kappa, mu, prec)
        assert rel(ctx.to_host(out, prec), W.twisted(U, phi, kappa, mu)) <= TOL[prec]
        e_in, e_out, tmp = ctx.halves(full, prec)[0], ctx.halves(out, prec)[0], ctx.empty_half(prec)
        for dagger, ref in ((False, W.schur), (True, W.schur_dag)):
            ctx.schur_apply(e_out, e_in, tmp, kappa, prec, dagger=dagger)
            assert rel(ctx.to_host(out, prec)[even], ref(U, half, kappa)[even]) <= TOL[prec]


@pytest.mark.parametrize("method", ["cg", "bicgstab"])
@pytest.mark.parametrize("inner,reals", [(F64, 18), (F32, 18), (F32, 12), (F16, 18), (F16, 12)])
@pytest.mark.parametrize("mu", [0.0, 0.03])
@pytest.mark.parametrize("mode", [0, 1])
def test_solves(method, inner, reals, mu, mode):
    dims = (8, 4, 4, 6)
    kappa = 0.12
    U, b = S.gauge_and_spinor(dims, 0.3, 5)
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        if inner != F64:
            ctx.gauge_upload(U, reals, inner)
        for p in {F64, inner}:
            ctx.set_launch(p, 1, 128, index_mode=mode)
        x = ctx.empty_full(F64)
        fn = ctx.cg_solve if method == "cg" else ctx.bicgstab_solve
        info = fn(x, ctx.to_device(b, F64), kappa, inner_prec=inner, mu=mu)
        xs = ctx.to_host(x, F64)
    res = np.linalg.norm(b - W.twisted(U, xs, kappa, mu)) / np.linalg.norm(b)
    assert res <= 1e-10, (res, info.as_dict())


def test_large_lattice_by_default():
    """Past the split kernel's range the library takes this kernel by itself."""
    dims = (16, 10, 12, 14)
    U, phi = S.gauge_and_spinor(dims, 0.3, 7)
    H = C.hopping(U, phi)
    with Context(dims) as ctx:
        for prec, reals in FORMATS[2:]:
            ctx.gauge_upload(U, reals, prec)
            got = gpu_hopping_full(ctx, phi, prec)
            assert rel(got, H) <= TOL[prec]
            ctx.set_launch(prec, 1, 128)
            assert np.array_equal(gpu_hopping_full(ctx, phi, prec), got)
            ctx.set_launch(prec, 1)


def test_debug_build_runs_clean():
    """The device bounds guards of this kernel: debug_battery_site_kernel.py through the debug library."""
    from paper_1405_0700_gb300 import _build

    env = dict(os.environ, PLQ_LIBRARY=_build.build(debug=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_battery_site_kernel.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert lines, r.stdout[-2000:] + r.stderr[-4000:]
    rep = json.loads(lines[-1])
    assert rep["library"].endswith("libplq_debug.so")
    assert rep["checks"] >= 40 and not rep["failures"], rep
    assert r.returncode == 0
