"""Branches of the element kernels that the small parity meshes do not reach: residual passes with
whole-warp element groups (meshes of two or more CTAs per SM, a last group that is not full), the
hexahedral block kernel of each degree, the embedded (EFR) block kernel of each degree, and fluxes
without viscosity.

The large meshes repeat one oracle-sized periodic tile of exactly representable spacing, with its
state and its implicit rows, so the residual of every copy is the tile's.  Tolerances are those of
the parity tests, for the same reason: FP64 arrays differ by the order of evaluation only (1e-11 of
the largest entry), FP32 blocks by the rounding of O(n) accumulated terms (3e-5)."""

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
from oracle.blocks import element_blocks  # noqa: E402
from oracle.efr import EmbeddedDiscretisation  # noqa: E402
from oracle.fr import Discretisation  # noqa: E402
from oracle.fr3d import Discretisation3D, element_blocks_3d  # noqa: E402
from oracle.physics import make_physics  # noqa: E402
from workloads import make_config  # noqa: E402
from workloads.mesh import BC_WALL, structured_hexes, structured_quads, tanh_nodes, uniform_nodes  # noqa: E402
from workloads.states import sample_points_hex  # noqa: E402

DEV = "cuda"
NS = {"kind": "ns", "gamma": 1.4, "mu": 5e-3, "Pr": 0.72, "lref": 1.0}
EDAC = {"kind": "edac", "theta": 100.0, "nu": 1e-3, "lref": 1.0}
ADVDIFF = {"kind": "advdiff", "beta": (1.0, 0.5), "nu": 0.01, "lref": 1.0}
NS3 = {"kind": "ns3d", "gamma": 1.4, "mu": 2e-2, "Pr": 0.72, "lref": 1.0}
BASE = {"ns": [1.0, 0.3, -0.2, 2.6], "edac": [0.1, 1.0, 0.4], "advdiff": [1.0], "ns3d": [1.0, 0.3, -0.2, 0.1, 2.6]}
TX, TY, COPIES = 9, 7, 9  # tile of 63 elements; 81 x 63 = 5103 elements: the last group is never full


def _tiled(phys, p, band, copies):
    """(mesh of copies x copies tiles, state): every tile with the same state and implicit rows."""
    nx, ny = TX * copies, TY * copies
    imp = None
    if band:
        rows = np.arange(ny) % TY
        imp = np.repeat((rows >= 2) & (rows < 5), nx)
    mesh = structured_quads(uniform_nodes(nx, 0, 0.25 * nx), uniform_nodes(ny, 0, 0.25 * ny), p=p, implicit=imp)
    base = np.asarray(BASE[phys["kind"]])
    one = base * (1 + 1e-2 * np.random.default_rng(p).standard_normal((TY, TX, (p + 1) ** 2, len(base))))
    return mesh, np.ascontiguousarray(np.tile(one, (copies, copies, 1, 1)).reshape(nx * ny, (p + 1) ** 2, len(base)))


RESIDUALS = [("advdiff", ADVDIFF, 1, True), ("ns", NS, 2, False), ("ns_band", NS, 2, True), ("edac", EDAC, 3, False),
             ("ns_band", NS, 3, True), ("ns_inviscid_band", dict(NS, mu=0.0), 3, True), ("ns", NS, 4, False),
             ("ns_band", NS, 5, True)]


def _rel(a, b):
    a = np.asarray(a, dtype=np.float64)
    b = np.asarray(b, dtype=np.float64)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


@pytest.mark.parametrize("phys,p,band", [r[1:] for r in RESIDUALS], ids=[f"{r[0]}_p{r[2]}" for r in RESIDUALS])
def test_residual_of_large_meshes(phys, p, band):
    tile, U1 = _tiled(phys, p, band, 1)
    d = Discretisation(tile, make_physics(phys))
    Ro, go = d.full_residual(U1, d.initial_trace(U1))
    mesh, U = _tiled(phys, p, band, COPIES)
    ctx = pkg.Context(mesh, phys)
    u = torch.tensor(U, device=DEV)
    R, g = ctx.fr_residual(u, ctx.hfr_initial_trace(u))
    want = np.tile(np.asarray(Ro).reshape(TY, TX, -1), (COPIES, COPIES, 1))
    assert _rel(R.cpu().numpy().reshape(want.shape), want) < 1e-11
    if phys["kind"] == "edac" or not phys.get("mu", 1.0):
        # u^ is the mean of both sides, where the convective parts of g cancel: what is left of 25 is
        # 2.5e-4 here (EDAC) or rounding alone (no viscosity), not an array to compare to 1e-11 of itself
        return
    # trace values have other positions in the large mesh: each occurs once per copy
    got = np.sort(g.cpu().numpy().reshape(-1))
    assert _rel(got, np.sort(np.tile(np.asarray(go).reshape(-1), COPIES**2))) < 1e-11
    ctx.close()


def _check_blocks(ctx, d, phys, U, make, trace, tol):
    uh = trace * (1 + 1e-3 * np.random.default_rng(1).standard_normal(trace.shape))
    flat = lambda x: torch.tensor(np.ascontiguousarray(x).reshape(-1), device=DEV)  # noqa: E731
    ctx.hfr_local_jacobian(flat(U), flat(uh), flat(U), 0.021)
    ref = make(d, U, uh, 0.021)
    for key, blk in zip("ABCD", ref):
        got = ctx.export_blocks(key)
        for k, e in enumerate(d.imp_idx):
            assert _rel(got[k], blk[e]) < tol, (key, e)
    ctx.close()


PREC = [(pkg.FR_PREC_FP64, 1e-11), (pkg.FR_PREC_FP32, 3e-5)]


@pytest.mark.parametrize("prec,tol", PREC, ids=["fp64", "fp32"])
@pytest.mark.parametrize("p,wall,mu", [(1, False, 2e-2), (1, True, 2e-2), (2, True, 2e-2), (2, False, 0.0), (3, False, 2e-2)])
def test_hex_blocks_of_each_degree(p, wall, mu, prec, tol):
    phys, n = dict(NS3, mu=mu), (2, 3, 2) if wall else (3, 3, 3)
    j = np.arange(n[0] * n[1] * n[2]) // n[0] % n[1]
    if wall:
        mesh = structured_hexes(uniform_nodes(2, 0, 2 * np.pi), tanh_nodes(3, 1.5), uniform_nodes(2, 0, np.pi), p=p,
                                periodic=(True, False, True), implicit=j != 1, bc_y=(BC_WALL, BC_WALL))
    else:
        mesh = structured_hexes(*[uniform_nodes(3, 0, 2.0)] * 3, periodic=(True, True, True), jitter=0.1, seed=6, p=p,
                                implicit=j != 2)
    x = sample_points_hex(mesh, p)
    U = np.asarray(BASE["ns3d"]) * (1 + 1e-2 * np.random.default_rng(p).standard_normal(x.shape[:2] + (5,)))
    ctx, d = pkg.Context(mesh, phys, precision=prec), Discretisation3D(mesh, make_physics(phys))
    _check_blocks(ctx, d, phys, U, element_blocks_3d, d.initial_trace(U), tol)


@pytest.mark.parametrize("prec,tol", PREC, ids=["fp64", "fp32"])
@pytest.mark.parametrize("p", [1, 4, 5])
def test_embedded_blocks_of_each_degree(p, prec, tol):
    w = make_config("vortex", n=4, p=p, jitter=0.1, seed=5, re=300.0)
    ctx = pkg.Context(w.mesh, w.physics, precision=prec, trace_kind=pkg.FR_TRACE_EFR)
    d = EmbeddedDiscretisation(w.mesh, make_physics(w.physics), None)
    _check_blocks(ctx, d, w.physics, np.asarray(w.u0), element_blocks, d.initial_trace(w.u0), tol)


def _grid(p, physics):
    """Periodic 5 x 4 quadrilaterals, degrees spread over p, all implicit: every face carries a trace."""
    deg = np.random.default_rng(3).choice(p, size=20).astype(np.int32)
    mesh = structured_quads(uniform_nodes(5, 0, 2.0), uniform_nodes(4, 0, 1.6), jitter=0.1, seed=2, p=deg)
    rng = np.random.default_rng(4)
    base = np.asarray(BASE[physics["kind"]])
    return mesh, physics, np.concatenate([(base * (1 + 1e-2 * rng.standard_normal(((q + 1) ** 2, len(base))))).reshape(-1) for q in deg])


def _hexes(p):
    mesh = structured_hexes(*[uniform_nodes(3, 0, 2.0)] * 3, periodic=(True, True, True), jitter=0.1, seed=6, p=p)
    rng = np.random.default_rng(p)
    return mesh, NS3, (np.asarray(BASE["ns3d"]) * (1 + 1e-2 * rng.standard_normal((27, (p + 1) ** 3, 5)))).reshape(-1)


# (mixed degrees with EDAC and the condensation of hexahedra of p = 1 are refused)
PRECOND = {"scalar_2_to_4": lambda: _grid([1, 2, 3], ADVDIFF), "ns_8_to_24": lambda: _grid([1, 2, 3, 5], NS),
           "hex_45": lambda: _hexes(2), "hex_80": lambda: _hexes(3)}


@pytest.mark.parametrize("prec,u", [(pkg.FR_PREC_FP64, 2.0**-53), (pkg.FR_PREC_FP32, 2.0**-24)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("name", list(PRECOND))
def test_face_block_inverses(name, prec, u):
    """The face-block inverses of general meshes against numpy's, from the same S: elimination with
    partial pivoting is within about 4 bs u cond of the inverse (largest entries compared)."""
    mesh, phys, U = PRECOND[name]()
    ctx = pkg.Context(mesh, phys, precision=prec)
    assert ctx.general
    us = torch.tensor(U, device=DEV).reshape(ctx.state_shape).contiguous()
    ctx.hfr_local_jacobian(us, ctx.hfr_initial_trace(us), us, 0.02)
    ctx.hfr_condense()
    S = [np.asarray(b, dtype=np.float64) for b in ctx.export_blocks("S")]
    got = ctx.hfr_export("Pinv").cpu().numpy().astype(np.float64)
    bs = np.diff(ctx.trace_off)
    P = [np.zeros((b, b)) for b in bs]
    for k, faces in enumerate(mesh.face_of):  # all implicit: traces are numbered as the faces
        lo = 0
        for t in faces:
            P[t] += S[k][lo:lo + bs[t], lo:lo + bs[t]]
            lo += bs[t]
    at = 0
    for t, Pt in enumerate(P):
        n = len(Pt)
        want, have = np.linalg.inv(Pt), got[at:at + n * n].reshape(n, n)
        assert _rel(have, want) < 4 * n * u * np.linalg.cond(Pt), (t, n)
        at += n * n
    assert at == got.size
    ctx.close()
