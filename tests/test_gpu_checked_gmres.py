"""The single-launch GMRES cycle of any layout in the bounds-checked build (FR_CHECKED): cycles of the
longest restart length address rows 0 .. 63 of the preconditioned basis only, on a uniform shape
(one cluster; the whole device), on walls and on EFR nodes, on the stream and in a stage graph, and
nothing is recorded.  The library runs in a child process of its own."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import json, sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
import paper_2401_16632_gb300 as pkg
pkg.load_library(sys.argv[1])
from workloads import make_config
out = {}

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
    ctx.hfr_local_jacobian(u, uh * 1.001, u * 0.999, scale * w.dt)
    ctx.hfr_condense()
    x, its, rel = ctx.hfr_trace_gmres(rtol=1e-11, maxit=3000)
    out[name] = {"its": its, "rel": rel, "status": list(pkg.fr_checked_status())}
    if name == "wall":  # the same cycle as the body of a captured stage
        ctx.imex_stage_set_graph(True)
        R_hist, us = ctx.empty(3, *ctx.state_shape), ctx.empty(*ctx.state_shape)
        ctx.imex_stage(0, w.dt, u, us, uh, R_hist)
        st = ctx.imex_stage(1, w.dt, u, us, uh, R_hist, newton_tol=1e-10, gmres_rtol=1e-11, gmres_maxit=3000)
        out["graph"] = {"its": st["gmres_iterations"] // max(st["newton_iterations"], 1), "rel": 0.0,
                        "status": list(pkg.fr_checked_status())}
    ctx.close()
print("RESULT " + json.dumps(out))
'''


@pytest.fixture(scope="module")
def run():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    from paper_2401_16632_gb300.build import build

    lib = build(checked=True)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD, lib], cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    line = [l for l in r.stdout.splitlines() if l.startswith("RESULT ")][-1]
    return json.loads(line[len("RESULT "):])


@pytest.mark.parametrize("name", ["cluster", "grid", "wall", "efr", "graph"])
def test_full_cycles_stay_inside_the_preconditioned_basis(run, name):
    assert run[name]["its"] > 64 and run[name]["rel"] <= 1e-10
    assert run[name]["status"] == [0, 0, 0]
