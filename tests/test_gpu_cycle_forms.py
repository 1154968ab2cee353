"""The single-launch GMRES cycle on both sides of the size (25 000 trace values) from which the second
Gram-Schmidt pass is made only where cancellation asks for it, against the cycle of short kernels on the
same condensed system: EFR nodes of p = 4 (28 values per element), at the usual step, where nearly every
column needs the pass, and at ten times it, where about half do without.

Tolerance: both solves end at a relative residual rtol, and the condition numbers are below 1e3 and (ten
times the step) 1e4: the solutions agree to 2 rtol times that.  FP32 blocks: a mat-vec carries about
1e-7, so rtol is 1e-6 and the usual step only."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2401_16632_gb300.build import build

    build()
    torch.cuda.set_device(0)


import paper_2401_16632_gb300 as pkg  # noqa: E402
from workloads import make_config  # noqa: E402


@pytest.mark.parametrize("n", [29, 30])  # 23 548 and 25 200 values
@pytest.mark.parametrize("prec,scale,rtol,cond", [(pkg.FR_PREC_FP64, 0.3, 1e-10, 1e3), (pkg.FR_PREC_FP64, 3.0, 1e-9, 1e4),
                                                  (pkg.FR_PREC_FP32, 0.3, 1e-6, 1e3)])
def test_both_sides_of_the_line(n, prec, scale, rtol, cond):
    w = make_config("vortex", n=n, p=4)
    ctx = pkg.Context(w.mesh, w.physics, precision=prec, trace_kind=pkg.FR_TRACE_EFR)
    assert (ctx.info.trace_values >= 25000) == (n == 30)
    u = torch.tensor(np.asarray(w.u0), device="cuda").reshape(ctx.state_shape).contiguous()
    uh = ctx.hfr_initial_trace(u)
    ctx.hfr_local_jacobian(u, uh * 1.001, u * 0.999, scale * w.dt)
    ctx.hfr_condense()
    a, ia, ra = ctx.hfr_trace_gmres(rtol=rtol, maxit=3000)
    a = a.clone()
    ctx.hfr_gmres_set_mode(pkg.FR_GMRES_SHORT)
    b, ib, rb = ctx.hfr_trace_gmres(rtol=rtol, maxit=3000)
    assert abs(ia - ib) <= 2 + ib // 10, (ia, ib)
    assert ra <= max(10 * rtol, 3 * rb)
    assert float((a - b).norm()) <= 2 * rtol * cond * float(b.norm())
    ctx.close()
