"""The single-launch GMRES cycle of any layout in the bounds-checked build (FR_CHECKED): cycles of the
longest restart length address rows 0 .. 63 of the preconditioned basis only, on a uniform shape
(one cluster; the whole device), on walls and on EFR nodes, on the stream and in a stage graph, and
nothing is recorded; a corrupted entry of either table that the cycle gathers through, planted through
the checked build's import, is caught (site, index) without a fault, and the normal build refuses that
import.  Each library runs in a child process of its own."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes, json, sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
import paper_2401_16632_gb300 as pkg
pkg.load_library(sys.argv[1])
from workloads import make_config
out = {}

def status():
    try:
        return list(pkg.fr_checked_status())
    except pkg.HfrError as e:
        return ["unsupported", e.code]

def context(w, trace=0):
    ctx = pkg.Context(w.mesh, w.physics, precision=pkg.FR_PREC_FP64, tableau=pkg.FR_TAB_SDIRK2, gmres_restart=64,
                      trace_kind=trace)
    u0 = ctx.pack_state(w.u0) if isinstance(w.u0, list) else np.asarray(w.u0)
    return ctx, torch.tensor(u0, device="cuda").reshape(ctx.state_shape).contiguous()

CASES = {"cluster": (lambda: make_config("advdiff8"), 30.0, 0),
         "grid": (lambda: make_config("advdiff", n=37, p=3, jitter=0.1, seed=2), 3.0, 0),
         "wall": (lambda: make_config("boundary_layer", nx=5, ny=60), 0.3, 0),
         "efr": (lambda: make_config("vortex", n=11, p=3), 3.0, pkg.FR_TRACE_EFR)}
for name, (make, scale, trace) in CASES.items():
    w = make()
    ctx, u = context(w, trace)
    uh = ctx.hfr_initial_trace(u)
    at_state = (u, uh * 1.001, u * 0.999, scale * w.dt)
    ctx.hfr_local_jacobian(*at_state)
    ctx.hfr_condense()
    x, its, rel = ctx.hfr_trace_gmres(rtol=1e-11, maxit=3000)
    out[name] = {"its": its, "rel": rel, "status": status()}
    if name == "wall":  # the same cycle as the body of a captured stage
        ctx.imex_stage_set_graph(True)
        R_hist, us = ctx.empty(3, *ctx.state_shape), ctx.empty(*ctx.state_shape)
        ctx.imex_stage(0, w.dt, u, us, uh, R_hist)
        st = ctx.imex_stage(1, w.dt, u, us, uh, R_hist, newton_tol=1e-10, gmres_rtol=1e-11, gmres_maxit=3000)
        out["graph"] = {"its": st["gmres_iterations"] // max(st["newton_iterations"], 1), "rel": 0.0,
                        "status": status()}
    if name == "wall":  # one entry of each gather table sent far out of range, then put back
        nT = int(np.sum(ctx.blk_nT))
        gmap = torch.full((nT,), -1, dtype=torch.int32, device="cuda")

        def table(call, which, t):
            return call(ctx.h, which, ctypes.c_void_p(t.data_ptr()), t.numel() * t.element_size())

        out["refused"] = [table(ctx.lib.hfr_export, 65, gmap), 0]
        vidx = torch.zeros((int((gmap >= 0).sum()),), dtype=torch.int64, device="cuda")
        out["refused"][1] = table(ctx.lib.hfr_export, 66, vidx) if out["refused"][0] == 0 else \
            table(ctx.lib.hfr_import, 66, torch.zeros(4, dtype=torch.int64, device="cuda"))
        if out["refused"][0] == 0:
            ctx.hfr_local_jacobian(*at_state)
            ctx.hfr_condense()
            for which, t, at in ((65, gmap, int(torch.nonzero(gmap >= 0)[7])), (66, vidx, 11)):
                bad = t.clone()
                bad[at] = 1 << 30
                pkg.fr_checked_status()
                assert table(ctx.lib.hfr_import, which, bad) == 0
                ctx.hfr_trace_gmres(rtol=1e-11, maxit=20, check=False)
                torch.cuda.synchronize()
                out[str(which)] = list(pkg.fr_checked_status())
                assert table(ctx.lib.hfr_import, which, t) == 0
            y, its2, rel2 = ctx.hfr_trace_gmres(rtol=1e-11, maxit=3000)
            out["restored"] = [its2 == its, float((y - x).norm()), list(pkg.fr_checked_status())]
    ctx.close()
print("RESULT " + json.dumps(out))
'''


def _run(lib):
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD, lib], cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    line = [l for l in r.stdout.splitlines() if l.startswith("RESULT ")][-1]
    return json.loads(line[len("RESULT "):])


@pytest.fixture(scope="module")
def run():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2401_16632_gb300.build import build

    return _run(build(checked=True))


@pytest.mark.parametrize("name", ["cluster", "grid", "wall", "efr", "graph"])
def test_full_cycles_stay_inside_the_preconditioned_basis(run, name):
    assert run[name]["its"] > 64 and run[name]["rel"] <= 1e-10
    assert run[name]["status"] == [0, 0, 0]


@pytest.mark.parametrize("table,site", [("65", 31), ("66", 35)])
def test_corrupted_gather_table_is_caught_without_a_fault(run, table, site):
    first, index, count = run[table]
    assert first == site and index == 1 << 30 and count >= 1


def test_restored_tables_solve_as_before(run):
    same_its, diff, status = run["restored"]
    assert same_its and diff == 0.0 and status == [0, 0, 0]


def test_normal_build_refuses_the_tables():
    from paper_2401_16632_gb300.build import build

    import paper_2401_16632_gb300 as pkg

    out = _run(build())
    assert out["refused"] == [pkg.FR_ERR_INVALID_ARG, pkg.FR_ERR_INVALID_ARG]
    assert "65" not in out
