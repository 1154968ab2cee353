"""The single-launch GMRES cycle of any trace layout against the cycle of short kernels
(hfr_gmres_set_mode(FR_GMRES_MULTI)) on the same condensed system: uniform shapes without a compiled
cycle, mixed degrees with walls, hexahedra, EFR nodes; systems small enough for one cluster and
larger ones on the whole device; restarts.

Tolerance: both solves end at a relative residual of 1e-11 (FP64) or 1e-6 (FP32 blocks, whose
mat-vec carries about 1e-7), and the condition numbers of these systems are below 1e3: the
solutions agree to 1e-8 and 1e-3."""

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

CASES = {
    "advdiff_p1": lambda: make_config("advdiff", n=3, p=1),
    "advdiff_p2": lambda: make_config("advdiff8"),
    "advdiff_p3_large": lambda: make_config("advdiff", n=37, p=3, jitter=0.1, seed=2),
    "edac_p2": lambda: make_config("edac", n=9, p=2),
    "edac_p4": lambda: make_config("edac", n=12, p=4, jitter=0.1),
    "vortex_p5": lambda: make_config("vortex", n=6, p=5, re=500.0),
    "wall_small": lambda: make_config("boundary_layer", nx=5, ny=60),
    "wall_large": lambda: make_config("boundary_layer", nx=60, ny=60),
    "hex_p2": lambda: make_config("channel3d", n=(4, 7, 3), p=2, layers=2),
    "hex_p3": lambda: make_config("channel3d", n=(3, 6, 4), p=3, layers=2),
    "efr_p3": lambda: make_config("vortex", n=11, p=3),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("prec", [pkg.FR_PREC_FP64, pkg.FR_PREC_FP32])
@pytest.mark.parametrize("restart", [30, 7])
def test_cycle_matches_short_kernels(name, prec, restart):
    w = CASES[name]()
    trace = pkg.FR_TRACE_EFR if name.startswith("efr") else pkg.FR_TRACE_HFR
    ctx = pkg.Context(w.mesh, w.physics, precision=prec, gmres_restart=restart, trace_kind=trace)
    u0 = ctx.pack_state(w.u0) if isinstance(w.u0, list) else np.asarray(w.u0)
    u = torch.tensor(u0, device="cuda").reshape(ctx.state_shape).contiguous()
    uh = ctx.hfr_initial_trace(u)
    ctx.hfr_local_jacobian(u, uh * 1.001, u * 0.999, 0.3 * w.dt)
    ctx.hfr_condense()
    rtol, tol = (1e-11, 1e-8) if prec == pkg.FR_PREC_FP64 else (1e-6, 1e-3)
    a, ia, ra = ctx.hfr_trace_gmres(rtol=rtol, maxit=3000)
    ctx.hfr_gmres_set_mode(pkg.FR_GMRES_MULTI)
    b, ib, rb = ctx.hfr_trace_gmres(rtol=rtol, maxit=3000)
    assert abs(ia - ib) <= 2 + ib // 10, (ia, ib)
    assert float((a - b).norm()) <= tol * float(b.norm())
    assert ra <= max(10 * rtol, 3 * rb)
