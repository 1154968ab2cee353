"""A NaN in an element block or in the Schur complement that a face block is summed from ends in a status
code or in NaN outputs, on every route of the condensation and of the face preconditioner: the pivot
searches take an unused row even where a column holds nothing but NaN, so that no row is left without
the step that its outputs are addressed by.  Clean blocks then condense bit for bit as before (no
tolerance)."""

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

SHAPES = [(9, 12), (36, 48), (64, 64), (100, 80), (144, 96)]


@pytest.mark.parametrize("prec", [pkg.FR_PREC_FP64, pkg.FR_PREC_FP32])
@pytest.mark.parametrize("spot", [(3, 5), (0, 0), (8, 8)])
def test_uneven_batch(prec, spot):
    dt = torch.float64 if prec == pkg.FR_PREC_FP64 else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    nA, nT = [s[0] for s in SHAPES for _ in (0, 1)], [s[1] for s in SHAPES for _ in (0, 1)]
    new = lambda *n: torch.randn(*n, generator=g, device="cuda", dtype=dt)  # noqa: E731
    A = [new(a, a) + 4 * a**0.5 * torch.eye(a, device="cuda", dtype=dt) for a in nA]
    nb = sum(a * t for a, t in zip(nA, nT))
    rest = new(nb), new(nb), new(sum(t * t for t in nT)), new(sum(nA)).double(), new(sum(nT)).double()
    pack = lambda blocks: torch.cat([a.reshape(-1) for a in blocks])  # noqa: E731
    good = pkg.hfr_condense_uneven(nA, nT, pack(A), *rest, precision=prec)
    ends = {"XB": [a * t for a, t in zip(nA, nT)], "S": [t * t for t in nT], "xr": nA, "t": nT, "piv": nA}
    for k in range(len(nA)):
        bad = [a.clone() for a in A]
        bad[k][spot] = float("nan")
        with pytest.raises(pkg.HfrError) as ei:
            pkg.hfr_condense_uneven(nA, nT, pack(bad), *rest, precision=prec)
        assert ei.value.code == pkg.FR_ERR_SINGULAR and ei.value.failed_element == k
    again = pkg.hfr_condense_uneven(nA, nT, pack(A), *rest, precision=prec)
    for name, n in ends.items():
        assert again[name].numel() == sum(n) and torch.equal(again[name], good[name])


CONTEXTS = {
    "advdiff_p1": lambda: make_config("advdiff", n=3, p=1),
    "advdiff_p2": lambda: make_config("advdiff8"),
    "advdiff_p3": lambda: make_config("advdiff", n=5, p=3),
    "edac_p2": lambda: make_config("edac", n=4, p=2),
    "edac_p4": lambda: make_config("edac", n=4, p=4),
    "vortex_p2": lambda: make_config("vortex", n=4, p=2, re=500.0),
    "vortex_p3": lambda: make_config("vortex", n=4, p=3, re=500.0),
    "vortex_p4": lambda: make_config("vortex", n=4, p=4, re=500.0),
    "vortex_p5": lambda: make_config("vortex", n=4, p=5, re=500.0),
    "wall": lambda: make_config("boundary_layer", nx=5, ny=60),
    "hex_p2": lambda: make_config("channel3d", n=(4, 7, 3), p=2, layers=2),
    "efr_p3": lambda: make_config("vortex", n=5, p=3),
}


@pytest.mark.parametrize("name", list(CONTEXTS))
@pytest.mark.parametrize("prec", [pkg.FR_PREC_FP64, pkg.FR_PREC_FP32])
def test_context(name, prec):
    w = CONTEXTS[name]()
    trace = pkg.FR_TRACE_EFR if name.startswith("efr") else pkg.FR_TRACE_HFR
    ctx = pkg.Context(w.mesh, w.physics, precision=prec, trace_kind=trace)
    u0 = ctx.pack_state(w.u0) if isinstance(w.u0, list) else np.asarray(w.u0)
    u = torch.tensor(u0, device="cuda").reshape(ctx.state_shape).contiguous()
    uh = ctx.hfr_initial_trace(u)
    ctx.hfr_local_jacobian(u, uh, u * 0.999, 0.3 * w.dt)
    blocks = {x: ctx.hfr_export(x).clone() for x in ("A", "D")}
    modes = [None]
    if prec == pkg.FR_PREC_FP32 and name in ("vortex_p2", "vortex_p3", "vortex_p4"):
        modes = [pkg.FR_CONDENSE_FMA, pkg.FR_CONDENSE_TENSOR_PRODUCTS, pkg.FR_CONDENSE_TENSOR]
    for mode in modes:
        if mode is not None:
            ctx.hfr_condense_set_mode(mode)
        ctx.hfr_condense()
        good = {x: ctx.hfr_export(x).clone() for x in ("S", "XB", "xr", "t", "Pinv")}
        for x in ("A", "D"):
            for spot in (0, 3, blocks[x].numel() // 2):
                bad = blocks[x].clone()
                bad.view(-1)[spot] = float("nan")
                ctx.hfr_import(x, bad)
                try:
                    ctx.hfr_condense()
                except pkg.HfrError as e:
                    assert e.code == pkg.FR_ERR_SINGULAR
                for y in ("XB", "xr") if x == "D" else ():  # D enters S alone
                    assert torch.equal(ctx.hfr_export(y), good[y])
                ctx.hfr_import(x, blocks[x])
        ctx.hfr_condense()
        for y, v in good.items():
            assert torch.equal(ctx.hfr_export(y), v), y
    ctx.close()
