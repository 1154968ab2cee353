"""hfr_gmres_set_mode / hfr_gmres_get_mode on contexts without a compiled cycle: setting the mode that
get returned changes nothing, FR_GMRES_SHORT gives the short kernels and FR_GMRES_MULTI the default
again; both forms of the cycle agree on the same condensed system.

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


def condensed(name, prec, restart, scale=0.3):
    w = CASES[name]()
    trace = pkg.FR_TRACE_EFR if name.startswith("efr") else pkg.FR_TRACE_HFR
    ctx = pkg.Context(w.mesh, w.physics, precision=prec, gmres_restart=restart, trace_kind=trace)
    u0 = ctx.pack_state(w.u0) if isinstance(w.u0, list) else np.asarray(w.u0)
    u = torch.tensor(u0, device="cuda").reshape(ctx.state_shape).contiguous()
    uh = ctx.hfr_initial_trace(u)
    ctx.hfr_local_jacobian(u, uh * 1.001, u * 0.999, scale * w.dt)
    ctx.hfr_condense()
    return ctx


def solve(ctx, rtol):
    n0 = ctx.kernel_launches()
    x, its, rel = ctx.hfr_trace_gmres(rtol=rtol, maxit=3000)
    return x.clone(), its, rel, ctx.kernel_launches() - n0


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("prec", [pkg.FR_PREC_FP64, pkg.FR_PREC_FP32])
@pytest.mark.parametrize("restart", [30, 7])
def test_modes_round_trip_and_both_forms_agree(name, prec, restart):
    ctx = condensed(name, prec, restart)
    rtol, tol = (1e-11, 1e-8) if prec == pkg.FR_PREC_FP64 else (1e-6, 1e-3)
    a, ia, ra, la = solve(ctx, rtol)
    assert ctx.hfr_gmres_get_mode() == pkg.FR_GMRES_MULTI
    ctx.hfr_gmres_set_mode(ctx.hfr_gmres_get_mode())
    b, ib, _, lb = solve(ctx, rtol)
    assert (ib, lb) == (ia, la) and torch.equal(a, b)
    with pytest.raises(pkg.HfrError) as ei:
        ctx.hfr_gmres_set_mode(pkg.FR_GMRES_FUSED)
    assert ei.value.code == pkg.FR_ERR_UNSUPPORTED
    ctx.hfr_gmres_set_mode(pkg.FR_GMRES_SHORT)
    assert ctx.hfr_gmres_get_mode() == pkg.FR_GMRES_SHORT
    c, ic, rc, lc = solve(ctx, rtol)
    assert lc >= 6 * ic  # a step: preconditioner, mat-vec, four Gram-Schmidt kernels at least
    assert abs(ia - ic) <= 2 + ic // 10, (ia, ic)
    assert float((a - c).norm()) <= tol * float(c.norm())
    assert ra <= max(10 * rtol, 3 * rc)
    ctx.hfr_gmres_set_mode(pkg.FR_GMRES_MULTI)
    d, i_d, _, ld = solve(ctx, rtol)
    assert (i_d, ld) == (ia, la) and torch.equal(a, d)


# a scale of the time step at which the solve takes more than 64 iterations: whole cycles of the
# longest restart length (and of one that is clamped to it).  The larger step raises the condition
# numbers to some 1e4: with both residuals at 1e-11 the solutions agree to 1e-6.
FULL = {"advdiff_p2": 30.0, "advdiff_p3_large": 3.0, "edac_p2": 3.0, "edac_p4": 3.0, "vortex_p5": 3.0, "wall_small": 0.3,
        "wall_large": 0.3, "hex_p2": 3.0, "hex_p3": 3.0, "efr_p3": 3.0}


@pytest.mark.parametrize("name", list(FULL))
def test_cycles_of_the_longest_restart_length(name):
    out = []
    for restart in (64, 100):
        ctx = condensed(name, pkg.FR_PREC_FP64, restart, FULL[name])
        out.append(solve(ctx, 1e-11))
    (a, ia, ra, la), (b, ib, _, lb) = out
    assert ia > 64 and (ia, la) == (ib, lb) and torch.equal(a, b)
    ctx.hfr_gmres_set_mode(pkg.FR_GMRES_SHORT)
    c, ic, rc, _ = solve(ctx, 1e-11)
    assert abs(ia - ic) <= 2 + ic // 10, (ia, ic)
    assert ra <= 1e-10 and rc <= 1e-10
    assert float((a - c).norm()) <= 1e-6 * float(c.norm())


@pytest.mark.parametrize("name", ["advdiff_p2", "edac_p2", "wall_small"])
def test_no_krylov_iteration_is_run_where_none_is_allowed(name):
    """imex_stage with gmres_maxit = 0: trace updates stay zero in both forms of the cycle."""
    w = CASES[name]()
    out = []
    for mode in (pkg.FR_GMRES_MULTI, pkg.FR_GMRES_SHORT):
        ctx = pkg.Context(w.mesh, w.physics, tableau=pkg.FR_TAB_SDIRK2)
        ctx.hfr_gmres_set_mode(mode)
        u0 = ctx.pack_state(w.u0) if isinstance(w.u0, list) else np.asarray(w.u0)
        u = torch.tensor(u0, device="cuda").reshape(ctx.state_shape).contiguous()
        uh = ctx.hfr_initial_trace(u)
        uh0 = uh.clone()
        R_hist, us = ctx.empty(3, *ctx.state_shape), ctx.empty(*ctx.state_shape)
        ctx.imex_stage(0, w.dt, u, us, uh, R_hist)
        with pytest.raises(pkg.HfrError) as ei:  # the trace equations are never solved
            ctx.imex_stage(1, w.dt, u, us, uh, R_hist, newton_tol=1e-12, newton_maxit=3, gmres_maxit=0)
        assert ei.value.code == pkg.FR_ERR_NOT_CONVERGED and ei.value.info.iteration == 3
        assert torch.equal(uh, uh0)
        out.append(us.clone())
    assert torch.equal(*out)


def test_large_uniform_fp64_systems_keep_the_short_kernels():
    """More than 10^8 values of S with faces of 24: the default is the short kernels' solve, bit for bit;
    one row of elements fewer and it is the single launch."""
    for n, short in ((105, True), (104, False)):  # 1.016 and 0.997 10^8 values
        w = make_config("vortex", n=n, p=5)
        ctx = pkg.Context(w.mesh, w.physics, precision=pkg.FR_PREC_FP64)
        u = torch.tensor(w.u0, device="cuda")
        uh = ctx.hfr_initial_trace(u)
        ctx.hfr_local_jacobian(u, uh * 1.001, u * 0.999, 0.3 * w.dt)
        ctx.hfr_condense()
        a, ia, _, la = solve(ctx, 1e-8)
        assert ctx.hfr_gmres_get_mode() == pkg.FR_GMRES_MULTI
        ctx.hfr_gmres_set_mode(pkg.FR_GMRES_SHORT)
        b, ib, _, lb = solve(ctx, 1e-8)
        assert (la == lb) == short
        if short:
            assert ia == ib and torch.equal(a, b)
        else:
            assert float((a - b).norm()) <= 1e-5 * float(b.norm())
        ctx.close()
