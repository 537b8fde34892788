"""Runs the one-thread-per-site operator kernel through the C ABI on ragged lattices, where the
library's own choice is the split kernel, and checks results against the oracle and the context's
device status word.  Started by test_gpu_site_kernel.py in a child process whose PLQ_LIBRARY names
the PLQ_DEBUG build (device bounds guards).  Prints one JSON line and exits 0 when every check passed.
"""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))


def main():
    import numpy as np
    import torch  # noqa: F401  (device memory)

    import synthetic as S
    from gpuhelp import TOL, gpu_hopping_full, rel
    from oracle import c_oracle as C
    from oracle import wilson as W
    from paper_1405_0700_gb300 import F16, F32, F64, Context
    from paper_1405_0700_gb300 import plq

    failures, checks = [], 0

    def check(name, ok, status):
        nonlocal checks
        checks += 1
        if not ok or status != plq.PLQ_OK:
            failures.append({"check": name, "ok": bool(ok), "status": int(status)})

    kappa = 0.12
    for dims in [(6, 2, 4, 2), (14, 6, 2, 10), (8, 8, 4, 4)]:
        U, phi = S.gauge_and_spinor(dims, 0.3, 31)
        H = W.hopping(U, phi)
        for prec, reals in [(F64, 18), (F64, 12), (F32, 18), (F32, 12), (F16, 18), (F16, 12)]:
            with Context(dims) as ctx:
                ctx.gauge_upload(U, reals, prec)
                for block, mode, spt in [(128, 0, 0), (64, 1, 0), (96, 0, 2)]:
                    ctx.set_launch(prec, 1, block, mode, sites_per_thread=spt)
                    check(f"hop {dims} {prec} {reals} {(block, mode, spt)}",
                          rel(gpu_hopping_full(ctx, phi, prec), H) <= TOL[prec], ctx.device_status())
    dims = (8, 4, 4, 6)
    U, b = S.gauge_and_spinor(dims, 0.3, 33)
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, F64)
        ctx.gauge_upload(U, 12, F32)
        ctx.gauge_upload(U, 12, F16)
        for p in (F64, F32, F16):
            ctx.set_launch(p, 1, 128)
        bd, x = ctx.to_device(b, F64), ctx.empty_full(F64)
        for fn in (ctx.cg_solve, ctx.bicgstab_solve):
            for inner in (F64, F32, F16):
                fn(x, bd, kappa, inner_prec=inner)
                res = np.linalg.norm(b - C.wilson(U, ctx.to_host(x, F64), kappa)) / np.linalg.norm(b)
                check(f"{fn.__name__} {inner}", res <= 1e-10, ctx.device_status())
    print(json.dumps({"library": plq.LIB_PATH, "checks": checks, "failures": failures}))
    return 0 if not failures else 1


if __name__ == "__main__":
    sys.exit(main())
