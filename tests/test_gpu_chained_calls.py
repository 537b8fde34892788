"""Operator calls launched dependent on one another: chains without synchronisation, mixed with
copies, with other streams and captured in a caller's graph give the bits of the same calls
waited for one by one."""
import numpy as np
import pytest

import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1405_0700_gb300 import F16, F32, F64, Context  # noqa: E402

KAPPA = 0.12


# lattices of a few blocks (several kernels of a chain fit the GPU at once) and of more than fit
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 8), (16, 12, 12, 12), (32, 16, 16, 16)])
@pytest.mark.parametrize("prec", [F64, F32, F16])
def test_chain_equals_calls_waited_for(dims, prec):
    U = S.gauge_field(dims, 0.3, 71)
    phi = S.gaussian_spinor(dims, 72)
    with Context(dims) as ctx:
        ctx.gauge_upload(U, 18, prec)
        start = ctx.to_device(phi, prec)
        full, out = torch.empty_like(start), torch.empty_like(start)
        tmp, half = ctx.empty_half(prec), ctx.empty_half(prec)
        other = torch.cuda.Stream()

        def chain(wait, streams):
            """Every buffer is read and written again by the calls two and three launches on."""
            main = torch.cuda.current_stream()

            def done():
                if wait:
                    torch.cuda.synchronize()

            full.copy_(start)
            e, o = ctx.halves(full, prec)
            e2, o2 = ctx.halves(out, prec)
            for k in range(6):
                ctx.schur_apply(e2, e, tmp, KAPPA, prec)
                done()
                ctx.schur_apply(e, e2, tmp, KAPPA, prec, dagger=True)
                done()
                ctx.hopping_eo(1, o2, e, prec)
                done()
                ctx.hopping_eo(0, e2, o2, prec)
                done()
                if streams:  # one call of the chain on another stream, between two copies
                    other.wait_stream(main)
                    with torch.cuda.stream(other):
                        half.copy_(e2)
                        ctx.schur_apply(e2, half, tmp, KAPPA, prec)
                        half.copy_(o2)
                    main.wait_stream(other)
                    o2.copy_(half)
                else:
                    half.copy_(e2)
                    done()
                    ctx.schur_apply(e2, half, tmp, KAPPA, prec)
                    done()
                ctx.wilson_apply(full, out, KAPPA / 8, prec)
                done()
            ctx.twisted_apply(out, full, KAPPA, 0.1, prec)
            done()

        def bits():
            torch.cuda.synchronize()
            return out.view(torch.uint8).cpu().numpy().copy()

        chain(True, False)
        want = bits()
        assert np.isfinite(ctx.to_host(out, prec)).all()
        for streams in (False, True):
            for _ in range(3):
                out.zero_()
                chain(False, streams)
                assert np.array_equal(bits(), want)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                chain(False, streams)
            for _ in range(3):
                out.zero_()
                graph.replay()
                assert np.array_equal(bits(), want)
