"""Performance cases: what a program that uses this library has it do, through its public calls.

Each case is a dict of plain values; `prepare` makes what such a program holds before the call (mesh,
context, states on the GPU), `run` is one pass of its inner loop, `work` the arithmetic and the bytes
the pass cannot do without, `exact` the same results in plain 64-bit torch.  Newton is driven to
1e-11 of its first residual, so a pass ends at the stage's own solution and not at a point that the
rounding of the linear solve picks.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2401_16632_gb300 as hfr

DEV = "cuda"
PRECISION = {"fp64": hfr.FR_PREC_FP64, "fp32": hfr.FR_PREC_FP32, "bf16": hfr.FR_PREC_BF16}
NEWTON = {"newton_tol": 1e-11, "newton_maxit": 40, "gmres_rtol": 1e-4, "gmres_maxit": 3000}
GAMMA = 1.4


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest run: 8x8 advection-diffusion, one backward-Euler step, all FP64; launches and
        # host round trips are its whole cost
        {"name": "advdiff_step_8x8_p2_fp64", "kind": "steps", "physics": "advdiff", "nx": 8, "ny": 8, "p": 2,
         "precision": "fp64", "tableau": "be", "jitter": 0.0, "band": 0, "keep": False, "steps": 1, "filter": False},
        # the explicit side of an IMEX run: the spatial residual alone, high degree, an implicit band in
        # a large explicit mesh with uneven side lengths
        {"name": "residual_203x177_p5", "kind": "residual", "physics": "ns", "nx": 203, "ny": 177, "p": 5,
         "precision": "fp64", "jitter": 0.15, "band": 36},
        # an ordinary implicit stage: 64x64 vortex, p = 3, mixed precision, run as one CUDA graph
        {"name": "stage_64x64_p3_fp32", "kind": "stage", "physics": "ns", "nx": 64, "ny": 64, "p": 3,
         "precision": "fp32", "jitter": 0.0, "graph": True},
        # the benchmark's stage: 256x256, p = 4, 6.55 M implicit unknowns, mixed precision, CUDA graph
        {"name": "stage_256x256_p4_fp32", "kind": "stage", "physics": "ns", "nx": 256, "ny": 256, "p": 4,
         "precision": "fp32", "jitter": 0.0, "graph": True},
        # the plain FP64 path of the same stage at the ordinary size, call by call on the stream
        {"name": "stage_64x64_p3_fp64", "kind": "stage", "physics": "ns", "nx": 64, "ny": 64, "p": 3,
         "precision": "fp64", "jitter": 0.0, "graph": False},
        # a whole IMEX step on a small ragged mesh: skewed cells, odd counts, an implicit band between
        # explicit elements with interface faces on both sides
        {"name": "imex_step_61x47_p2_fp32", "kind": "steps", "physics": "ns", "nx": 61, "ny": 47, "p": 2,
         "precision": "fp32", "tableau": "sdirk2", "jitter": 0.15, "band": 13, "keep": False, "steps": 1, "filter": False},
        # the linearised operator for a caller's own trace solver: element blocks, condensation, and the
        # Schur complements, X_B and face preconditioner handed over
        {"name": "operator_64x64_p4_fp32", "kind": "operator", "physics": "ns", "nx": 64, "ny": 64, "p": 4,
         "precision": "fp32", "jitter": 0.15},
        # near-wall stage on a stretched mesh: p = 2..5 per element, wall and far field, CUDA graph
        {"name": "wall_stage_200x250_fp32", "kind": "wall", "nx": 200, "ny": 250, "precision": "fp32", "graph": True},
        # three-dimensional channel: hexahedra with implicit layers on both walls, CUDA graph
        {"name": "channel_stage_32x16x24_p3_fp32", "kind": "channel", "nx": 32, "ny": 16, "nz": 24, "p": 3,
         "layers": 3, "precision": "fp32", "graph": True},
        # the embedded variant (continuous trace) of the vortex stage, call by call on the stream
        {"name": "efr_stage_128x128_p4_fp32", "kind": "efr", "physics": "ns", "nx": 128, "ny": 128, "p": 4,
         "precision": "fp32", "jitter": 0.0, "graph": False},
        # artificial-compressibility run: four steps with the Jacobian kept, then the modal filter
        {"name": "edac_keep_4_steps_48x45_p3_fp32", "kind": "steps", "physics": "edac", "nx": 48, "ny": 45, "p": 3,
         "precision": "fp32", "tableau": "sdirk2", "jitter": 0.1, "band": 0, "keep": True, "steps": 4, "filter": True},
        # condensation of a batch of blocks of mixed degree, formed by the caller, FP64
        {"name": "uneven_condense_3000_fp64", "kind": "uneven", "n": 3000, "precision": "fp64"},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the listed kinds; sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(["advdiff", "residual", "stage", "stage", "stage64", "imex", "operator", "wall", "channel",
                       "efr", "edac", "uneven"])
    skew = rng.choice([0.0, 0.1, 0.15])
    if kind == "advdiff":
        return {"kind": "steps", "physics": "advdiff", "nx": _log(rng, 5, 40), "ny": _log(rng, 5, 40),
                "p": rng.choice([1, 2, 3]), "precision": "fp64", "tableau": rng.choice(["be", "sdirk2"]),
                "jitter": skew, "band": 0, "keep": False, "steps": 1, "filter": False}
    if kind == "residual":
        return {"kind": "residual", "physics": "ns", "nx": _log(rng, 8, 220), "ny": _log(rng, 8, 220),
                "p": rng.choice([2, 3, 4, 5]), "precision": "fp64", "jitter": skew, "band": rng.choice([0, 3, 8])}
    if kind == "stage":
        return {"kind": "stage", "physics": "ns", "nx": _log(rng, 12, 140), "ny": _log(rng, 12, 140),
                "p": rng.choice([2, 3, 4]), "precision": rng.choice(["fp32", "fp32", "fp32", "bf16"]),
                "jitter": skew, "graph": rng.random() < 0.7}
    if kind == "stage64":
        return {"kind": "stage", "physics": "ns", "nx": _log(rng, 8, 48), "ny": _log(rng, 8, 48),
                "p": rng.choice([2, 3, 4]), "precision": "fp64", "jitter": skew, "graph": False}
    if kind == "imex":
        ny = _log(rng, 12, 90)
        return {"kind": "steps", "physics": "ns", "nx": _log(rng, 8, 90), "ny": ny, "p": rng.choice([2, 3, 4]),
                "precision": "fp32", "tableau": rng.choice(["be", "sdirk2"]), "jitter": skew, "band": max(2, ny // 4),
                "keep": False, "steps": 1, "filter": False}
    if kind == "operator":
        return {"kind": "operator", "physics": "ns", "nx": _log(rng, 10, 90), "ny": _log(rng, 10, 90),
                "p": rng.choice([2, 3, 4]), "precision": "fp32", "jitter": skew}
    if kind == "wall":
        return {"kind": "wall", "nx": _log(rng, 16, 220), "ny": _log(rng, 70, 260), "precision": "fp32",
                "graph": rng.random() < 0.5}
    if kind == "channel":
        return {"kind": "channel", "nx": _log(rng, 4, 24), "ny": _log(rng, 8, 20), "nz": _log(rng, 3, 20),
                "p": rng.choice([2, 3]), "layers": rng.choice([2, 3]), "precision": "fp32",
                "graph": rng.random() < 0.5}
    if kind == "efr":
        return {"kind": "efr", "physics": "ns", "nx": _log(rng, 12, 120), "ny": _log(rng, 12, 120),
                "p": rng.choice([2, 3, 4]), "precision": "fp32", "jitter": skew, "graph": rng.random() < 0.5}
    if kind == "edac":
        return {"kind": "steps", "physics": "edac", "nx": _log(rng, 12, 60), "ny": _log(rng, 12, 60),
                "p": rng.choice([2, 3, 4]), "precision": "fp32", "tableau": "sdirk2", "jitter": skew, "band": 0,
                "keep": True, "steps": rng.choice([2, 3, 4]), "filter": True}
    return {"kind": "uneven", "n": _log(rng, 50, 4000), "precision": "fp64"}


# ----------------------------------------------------------------------------------------- meshes
class Mesh:
    """Corner coordinates and connectivity of a structured mesh, as `hfr.Context` takes them."""

    def __init__(self, nodes, cells, periodic, p, implicit, bc=None):
        d = len(cells)
        self.dim = d
        E = int(np.prod(cells))
        idx = np.stack(np.unravel_index(np.arange(E), cells[::-1])[::-1], axis=1)  # (E, d), first axis fastest
        corner = []
        for k in range(2**d):
            at = idx + [(k >> r) & 1 for r in range(d)]
            corner.append(nodes[tuple(at.T)])
        self.verts = np.stack(corner, axis=1)
        self.nbr = np.full((E, 2 * d), -1, np.int32)
        self.nbr_face = np.full((E, 2 * d), -1, np.int32)
        self.bc = np.zeros((E, 2 * d), np.int32)
        for r in range(d):
            for side in (0, 1):
                f, at = 2 * r + side, idx.copy()
                at[:, r] += 2 * side - 1
                inside = (at[:, r] >= 0) & (at[:, r] < cells[r])
                at[:, r] %= cells[r]
                e = np.ravel_multi_index(at[:, ::-1].T, cells[::-1])
                has = inside | periodic[r]
                self.nbr[has, f] = e[has]
                self.nbr_face[has, f] = f ^ 1
                if bc is not None:
                    self.bc[~has, f] = bc[f]
        own = np.arange(E * 2 * d).reshape(E, 2 * d)
        other = np.where(self.nbr >= 0, self.nbr.astype(np.int64) * 2 * d + self.nbr_face, own)
        first = np.minimum(own, other)  # faces numbered by their first appearance
        self.face_of = np.unique(first.reshape(-1), return_inverse=True)[1].reshape(E, 2 * d).astype(np.int32)
        self.implicit = implicit if implicit is not None else np.ones(E, bool)
        self.p = np.broadcast_to(np.asarray(p, np.int32), (E,))

    def points(self, x):
        """Images of the tensor product of the 1D points x, first axis fastest: (E, points, d)."""
        d, n = self.dim, len(x)
        at = np.stack([g.reshape(-1) for g in np.meshgrid(*[x] * d, indexing="ij")][::-1], axis=1)
        N = np.ones((n**d, 2**d))
        for k in range(2**d):
            for r in range(d):
                N[:, k] *= 0.5 * (1 + (2 * ((k >> r) & 1) - 1) * at[:, r])
        return np.einsum("sk,ekd->esd", N, self.verts)


def _quads(case, rng, side):
    """Periodic nx x ny quads on [0, side]^2; inner nodes moved by `jitter` of the spacing; `band` > 0
    makes only that many middle rows implicit."""
    nx, ny = case["nx"], case["ny"]
    X = np.stack(np.meshgrid(np.linspace(0, side, nx + 1), np.linspace(0, side, ny + 1), indexing="ij"), axis=-1)
    if case["jitter"]:
        d = rng.uniform(-case["jitter"], case["jitter"], X.shape) * [side / nx, side / ny]
        d[nx], d[:, ny] = d[0], d[:, 0]
        d[nx, ny] = d[0, 0]
        X = X + d
    imp = None
    if case.get("band"):
        j, lo = np.arange(nx * ny) // nx, (ny - case["band"]) // 2
        imp = (j >= lo) & (j < lo + case["band"])
    return Mesh(X, (nx, ny), (True, True), case["p"], imp)


def _gauss(p):
    return np.polynomial.legendre.leggauss(p + 1)[0]


def _energy(rho, v, pressure):
    return pressure / (GAMMA - 1.0) + 0.5 * rho * sum(c * c for c in v)


def _periodic_problem(case, seed):
    """(mesh, physics, state, dt) of the periodic quadrilateral cases."""
    rng = np.random.default_rng([seed, 1])
    p, kind = case["p"], case["physics"]
    side = 1.0 if kind == "advdiff" else 10.0
    mesh = _quads(case, rng, side)
    x, y = np.moveaxis(mesh.points(_gauss(p)), -1, 0) - 0.5 * side
    h = side / max(case["nx"], case["ny"])
    if kind == "advdiff":  # a Gaussian pulse about a point near the middle
        c = rng.uniform(-0.05, 0.05, 2)
        u = np.exp(-50.0 * ((x - c[0]) ** 2 + (y - c[1]) ** 2))[..., None]
        return mesh, {"kind": "advdiff", "beta": (1.0, 0.5), "nu": 0.01, "lref": 1.0}, u, 0.4 * h
    r2 = x * x + y * y
    if kind == "edac":  # a weak vortex carried by a uniform stream, with its balancing pressure
        amp = np.exp(0.5 * (1.0 - r2)) / (2 * np.pi)
        u = np.stack([-np.exp(1.0 - r2) / (8 * np.pi**2), 1.0 - amp * y, amp * x], axis=-1)
        u += rng.uniform(-1e-3, 1e-3, u.shape)
        dt = 4.0 * h / ((1.5 + math.sqrt(100.25)) * (2 * p + 1))
        return mesh, {"kind": "edac", "theta": 100.0, "nu": 1e-3, "lref": 1.0}, u, dt
    # isentropic vortex at M = 0.5 with 1e-3 noise; ten times the explicit step, half of it where
    # explicit elements take part
    mach, amp = 0.5, 5.0 / (2 * np.pi) * np.exp(0.5 * (1.0 - r2))
    vx, vy = mach - amp * y, amp * x
    T = 1 / GAMMA - (GAMMA - 1) * 25.0 / (8 * GAMMA * np.pi**2) * np.exp(1.0 - r2)
    rho = (T * GAMMA) ** (1 / (GAMMA - 1))
    u = np.stack([rho, rho * vx, rho * vy, _energy(rho, (vx, vy), rho * T)], axis=-1)
    u += rng.uniform(-1e-3, 1e-3, u.shape)
    cfl = 10.0 if not case.get("band") else 0.5
    return mesh, {"kind": "ns", "gamma": GAMMA, "mu": 5e-5, "Pr": 0.72, "lref": 1.0}, u, cfl * h / (1.5 * (2 * p + 1))


def _wall_problem(case, seed):
    """Stretched wall band: rows from 1e-5 growing by 1.15 up to square 1e-2 cells, wall below, far field
    above, degrees 2..5 spread at random, the lowest fifth of the rows implicit, a noisy free stream."""
    rng = np.random.default_rng([seed, 2])
    nx, ny, dx = case["nx"], case["ny"], 1e-2
    yn = np.concatenate([[0.0], np.cumsum(np.minimum(1e-5 * 1.15 ** np.arange(ny), dx))])
    X = np.stack(np.meshgrid(np.linspace(0, nx * dx, nx + 1), yn, indexing="ij"), axis=-1)
    imp = np.arange(nx * ny) // nx < round(0.2 * ny)
    deg = np.random.default_rng([nx, ny]).integers(2, 6, nx * ny)  # a mesh's degrees belong to the mesh
    mesh = Mesh(X, (nx, ny), (True, False), deg, imp, bc=(0, 0, hfr.FR_BC_WALL, hfr.FR_BC_FARFIELD))
    mach = 0.2
    u_inf = np.array([1.0, mach, 0.0, _energy(1.0, (mach,), 1 / GAMMA)])
    u = u_inf + rng.uniform(-1e-3, 1e-3, (int(np.sum((deg + 1) ** 2)), 4))
    phys = {"kind": "ns", "gamma": GAMMA, "mu": mach / 1.7e6, "Pr": 0.72, "lref": 1.0, "u_inf": u_inf}
    return mesh, phys, u.reshape(-1), dx / ((mach + 1.0) * 11)


def _channel_problem(case, seed):
    """Channel [0, 2 pi] x [-1, 1] x [0, pi], cells clustered to the walls at y = -1, 1, a
    Taylor-Green-like field of M = 0.1 shifted along the periodic axes; implicit wall layers."""
    rng = np.random.default_rng([seed, 3])
    nx, ny, nz, p = case["nx"], case["ny"], case["nz"], case["p"]
    yn = np.tanh(2.5 * (2 * np.arange(ny + 1) / ny - 1)) / np.tanh(2.5)
    axes = np.linspace(0, 2 * np.pi, nx + 1), yn, np.linspace(0, np.pi, nz + 1)
    X = np.stack(np.meshgrid(*axes, indexing="ij"), axis=-1)
    j = np.arange(nx * ny * nz) // nx % ny
    imp = (j < case["layers"]) | (j >= ny - case["layers"])
    wall = hfr.FR_BC_WALL
    mesh = Mesh(X, (nx, ny, nz), (True, False, True), p, imp, bc=(0, 0, wall, wall, 0, 0))
    x, y, z = np.moveaxis(mesh.points(_gauss(p)), -1, 0)
    mach, sx, sz = 0.1, *rng.uniform(0, np.pi, 2)
    damp = mach * (1 - y * y)
    vx = damp * np.sin(x + sx) * np.cos(y) * np.cos(2 * (z + sz))
    vy = -damp * np.cos(x + sx) * np.sin(y) * np.cos(2 * (z + sz))
    one = np.ones_like(x)
    u = np.stack([one, vx, vy, 0 * x, _energy(one, (vx, vy), 1 / GAMMA)], axis=-1)
    dt = min(2 * np.pi / nx, np.pi / nz) / ((mach + 1.0) * (2 * p + 1))
    return mesh, {"kind": "ns3d", "gamma": GAMMA, "mu": mach / 1.6e3, "Pr": 0.72, "lref": 1.0}, u.reshape(-1), dt


def _uneven_problem(case, seed):
    """Blocks of degrees 2..5 in equal numbers (nA = 4 (p + 1)^2, nT = 16 (p + 1)), in random order, packed one element
    after another; A is well away from singular, as I - a dt dR/du is."""
    deg = np.random.default_rng([seed, 4]).permutation(np.arange(case["n"]) % 4 + 2)
    nA, nT = (4 * (deg + 1) ** 2).tolist(), (16 * (deg + 1)).tolist()
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    new = lambda n: torch.randn(n, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    A = [new(a * a).view(a, a) / a**0.5 for a in nA]
    for a in A:
        a.diagonal().add_(4.0)
    nb = sum(a * t for a, t in zip(nA, nT))
    blocks = (torch.cat([a.reshape(-1) for a in A]), new(nb), new(nb), new(sum(t * t for t in nT)), new(sum(nA)), new(sum(nT)))
    return nA, nT, blocks


# ---------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    if case["kind"] == "uneven":
        nA, nT, blocks = _uneven_problem(case, seed)
        return {"case": case, "nA": nA, "nT": nT, "blocks": blocks}
    problem = {"wall": _wall_problem, "channel": _channel_problem}.get(case["kind"], _periodic_problem)
    mesh, physics, u, dt = problem(case, seed)
    tableau = hfr.FR_TAB_BE if case.get("tableau") == "be" else hfr.FR_TAB_SDIRK2
    trace = hfr.FR_TRACE_EFR if case["kind"] == "efr" else hfr.FR_TRACE_HFR
    ctx = hfr.Context(mesh, physics, precision=PRECISION[case["precision"]], tableau=tableau, trace_kind=trace)
    if case.get("graph"):
        ctx.imex_stage_set_graph(True)
    if case.get("keep"):
        ctx.imex_set_jacobian_policy(hfr.FR_JAC_KEEP)
    u = torch.as_tensor(u, dtype=torch.float64, device=DEV).reshape(ctx.state_shape).contiguous()
    uhat = ctx.hfr_initial_trace(u)
    return {"case": case, "ctx": ctx, "dt": dt, "u0": u, "uhat0": uhat, "u": u.clone(), "uhat": uhat.clone(),
            "R_hist": ctx.empty(ctx.info.nstages + 1, *ctx.state_shape), "u_stage": ctx.empty(*ctx.state_shape)}


def run(state):
    case = state["case"]
    if case["kind"] == "uneven":
        return hfr.hfr_condense_uneven(state["nA"], state["nT"], *state["blocks"], precision=PRECISION[case["precision"]])
    ctx, dt, u, uhat = state["ctx"], state["dt"], state["u"], state["uhat"]
    if case["kind"] == "residual":
        return ctx.fr_residual(state["u0"], state["uhat0"])
    if case["kind"] == "operator":
        ctx.hfr_local_jacobian(state["u0"], state["uhat0"], state["u0"], (1 - 0.5**0.5) * dt)
        ctx.hfr_condense()
        return {k: ctx.hfr_export(k) for k in ("S", "XB", "Pinv")}
    uhat.copy_(state["uhat0"])  # each pass starts from the same trace and state
    if case["kind"] == "steps":
        u.copy_(state["u0"])
        ctx.imex_steps(case["steps"], dt, u, uhat, refresh_every=100 if case["keep"] else 0, **NEWTON)
        if case["filter"]:
            ctx.fr_modal_filter(u, 36.0, 4.0, case["p"])
        return u, uhat
    R, u_stage = state["R_hist"], state["u_stage"]
    ctx.imex_stage(0, dt, state["u0"], u_stage, uhat, R, **NEWTON)
    ctx.imex_stage(1, dt, state["u0"], u_stage, uhat, R, **NEWTON)
    return u_stage, uhat, R[:2]


# ------------------------------------------------------------------------------------------- work
def _condense_flops(nA, nT):
    """LU of A, X = A^-1 [B | r], D - C X_B and s - C x_r."""
    return 2 / 3 * nA**3 + 2.0 * nA * nA * (nT + 1) + 2.0 * nT * nA * (nT + 1)


def work(case):
    kind = case["kind"]
    size = 8 if case["precision"] == "fp64" else 4
    if kind == "uneven":  # inputs A, B, C, D, r, s; outputs LU, X_B, S, piv, x_r, t
        b = f = 0.0
        for p in (2, 3, 4, 5):
            nA, nT = 4 * (p + 1) ** 2, 16 * (p + 1)
            b += (2 * nA * nA + 3 * nA * nT + 2 * nT * nT + 2 * (nA + nT)) * size + 4 * nA
            f += _condense_flops(nA, nT)
        return {"bytes": b * case["n"] / 4, "flops": f * case["n"] / 4}
    if kind == "wall":
        E, shapes = case["nx"] * case["ny"], [(4 * (p + 1) ** 2, 16 * (p + 1)) for p in (2, 3, 4, 5)]
        frac, d = round(0.2 * case["ny"]) / case["ny"], 2
    elif kind == "channel":
        n = case["p"] + 1
        E, shapes, frac, d = case["nx"] * case["ny"] * case["nz"], [(5 * n**3, 30 * n * n)], 2 * case["layers"] / case["ny"], 3
    else:
        n, nv = case["p"] + 1, {"advdiff": 1, "edac": 3, "ns": 4}[case["physics"]]
        E, shapes, frac, d = case["nx"] * case["ny"], [(nv * n * n, 4 * nv * n)], 1.0, 2
        if case.get("band"):
            frac = case["band"] / case["ny"]
    mean = lambda g: sum(g(a, t) for a, t in shapes) / len(shapes)  # noqa: E731
    nA, nT = mean(lambda a, t: a), mean(lambda a, t: t)
    point = 60.0 * d  # fluxes at a point, and its line sums
    trace = 0.5 * frac * E * nT
    if kind == "residual":  # u, u^ and the metrics in, R and g out
        return {"bytes": 8.0 * E * (2 * nA + 5 * nA / 4 + 3 * nT / 4) + 16.0 * trace, "flops": point * E * (nA + nT)}
    solve = frac * E * mean(_condense_flops)
    if kind == "operator":  # u, u^ in, S, X_B and the face inverses out
        out = E * (nT * nT + nA * nT + nT * nT / 8) * size
        return {"bytes": 8.0 * (E * nA + trace) + out, "flops": solve + 2.0 * E * (nA + nT) ** 2}
    # a stage: three Newton iterations of about 15 Krylov iterations; u, u^ in, u, u^, R out
    stages = case.get("steps", 1) * (2 if case.get("tableau") == "sdirk2" else 1)
    lin = 1 if case.get("keep") else 3 * stages
    krylov = 2.0 * frac * E * mean(lambda a, t: t * t) * 45 * stages
    io = 8.0 * (4 * E * nA + 2 * trace)
    return {"bytes": io, "flops": lin * (solve + 2.0 * frac * E * mean(lambda a, t: (a + t) ** 2)) + krylov + 5 * stages * point * E * (nA + nT)}


# ------------------------------------------------------------------------------------------ exact
class Plain:
    """The hybridized flux-reconstruction operator on periodic quadrilaterals in 64-bit torch."""

    def __init__(self, mesh, phys):
        t = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=DEV)  # noqa: E731
        self.ph, p = phys, int(mesh.p[0])
        n = self.n = p + 1
        x, w = np.polynomial.legendre.leggauss(n)
        V = np.polynomial.legendre.legvander(x, p)
        dV = np.stack([np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c)) for c in np.eye(n)], axis=1)
        ends = np.polynomial.legendre.legvander(np.array([-1.0, 1.0]), p)
        Vi = np.linalg.inv(V)
        self.D, L = t(dV @ Vi), ends @ Vi
        self.V, self.Vi = V, Vi
        self.end = t(L)
        self.lift1 = t(np.stack([-L[0] / w, L[1] / w]))  # derivatives of the correction functions
        self.w = t(w)
        E = mesh.verts.shape[0]
        self.E, self.imp = E, t(mesh.implicit)
        self.nbr, self.nbf = t(mesh.nbr.astype(np.int64)), t(mesh.nbr_face.astype(np.int64))

        def metric(xi, eta):  # adjugate rows S[r] = J grad xi_r at reference points
            c = mesh.verts
            gx = [0.25 * s * (1 + q * eta) for s, q in ((-1, -1), (1, -1), (-1, 1), (1, 1))]
            ge = [0.25 * q * (1 + s * xi) for s, q in ((-1, -1), (1, -1), (-1, 1), (1, 1))]
            dx = np.einsum("ks,ekd->esd", np.array(gx), c)
            de = np.einsum("ks,ekd->esd", np.array(ge), c)
            S = np.stack([np.stack([de[..., 1], -de[..., 0]], -1), np.stack([-dx[..., 1], dx[..., 0]], -1)], axis=-2)
            return S, dx[..., 0] * de[..., 1] - de[..., 0] * dx[..., 1]

        S, J = metric(np.tile(x, n), np.repeat(x, n))
        self.S, self.J = t(S), t(J)
        N = []
        for f in range(4):
            r, sg = f >> 1, 2 * (f & 1) - 1.0
            one = np.full(n, sg)
            N.append(sg * metric(*((one, x) if r == 0 else (x, one)))[0][..., r, :])
        N = np.stack(N, axis=1)  # (E, 4, n, 2)
        Jf = np.linalg.norm(N, axis=-1)
        self.Jf, self.nrm = t(Jf), t(N / Jf[..., None])
        both, one = mesh.implicit[:, None] & mesh.implicit[mesh.nbr], mesh.implicit[:, None] != mesh.implicit[mesh.nbr]
        self.trace, self.imex = t(both)[..., None, None], t(one)[..., None, None]
        ids = np.unique(mesh.face_of[both])
        of = np.full(int(mesh.face_of.max()) + 1, -1)
        of[ids] = np.arange(len(ids))
        self.tr = t(np.where(both, of[mesh.face_of], len(ids)))  # (E, 4), off traces: one past the end
        self.ntrace = len(ids)
        self.nv = {"advdiff": 1, "edac": 3, "ns": 4}[phys["kind"]]

    # ---- physics: fluxes (..., 2, nv), wave speed and stabilisation
    def conv(self, u):
        ph = self.ph
        if ph["kind"] == "advdiff":
            return torch.stack([ph["beta"][0] * u, ph["beta"][1] * u], -2)
        if ph["kind"] == "edac":
            P, vx, vy = u.unbind(-1)
            Pt = P + ph["theta"]
            return torch.stack([torch.stack([vx * Pt, vx * vx + P, vx * vy], -1), torch.stack([vy * Pt, vy * vx, vy * vy + P], -1)], -2)
        rho, mx, my, En = u.unbind(-1)
        vx, vy = mx / rho, my / rho
        pr = (GAMMA - 1) * (En - 0.5 * (mx * vx + my * vy))
        return torch.stack([torch.stack([mx, mx * vx + pr, mx * vy, (En + pr) * vx], -1),
                            torch.stack([my, my * vx, my * vy + pr, (En + pr) * vy], -1)], -2)

    def visc(self, u, q):
        ph = self.ph
        if ph["kind"] != "ns":
            return ph["nu"] * q
        rho, mx, my, En = (c[..., None] for c in u.unbind(-1))
        vx, vy = mx / rho, my / rho
        dvx, dvy = (q[..., 1] - vx * q[..., 0]) / rho, (q[..., 2] - vy * q[..., 0]) / rho
        dT = (GAMMA - 1) * ((q[..., 3] - En / rho * q[..., 0]) / rho - vx * dvx - vy * dvy)
        mu = ph["mu"]
        dil = 2 / 3 * (dvx[..., 0] + dvy[..., 1])
        xx, yy, xy = mu * (2 * dvx[..., 0] - dil), mu * (2 * dvy[..., 1] - dil), mu * (dvx[..., 1] + dvy[..., 0])
        vx, vy, k = vx[..., 0], vy[..., 0], mu * GAMMA / ((GAMMA - 1) * ph["Pr"])
        o = torch.zeros_like(xx)
        return torch.stack([torch.stack([o, xx, xy, vx * xx + vy * xy + k * dT[..., 0]], -1),
                            torch.stack([o, xy, yy, vx * xy + vy * yy + k * dT[..., 1]], -1)], -2)

    def speed(self, u, stab):
        ph, nx, ny = self.ph, self.nrm[..., 0], self.nrm[..., 1]
        if ph["kind"] == "advdiff":
            a = (ph["beta"][0] * nx + ph["beta"][1] * ny).abs() + 0 * u[..., 0]
            return a + ph["nu"] / ph["lref"] if stab else a
        if ph["kind"] == "edac":
            P, vx, vy = u.unbind(-1)
            v2 = vx * vx + vy * vy if stab else (vx * nx + vy * ny) ** 2
            a = 1.5 * v2.sqrt() + (0.25 * v2 + P + ph["theta"]).sqrt()
            return a + ph["nu"] / ph["lref"] if stab else a
        rho, mx, my, En = u.unbind(-1)
        pr = (GAMMA - 1) * (En - 0.5 * (mx * mx + my * my) / rho)
        a = ((mx * nx + my * ny) / rho).abs() + (GAMMA * pr / rho).sqrt()
        return a + ph["mu"] / (rho * ph["lref"]) if stab else a

    # ---- operator
    def faces(self, X):  # (E, ns, ...) -> values at the points of the four faces (E, 4, n, ...)
        G = X.reshape(self.E, self.n, self.n, *X.shape[2:])
        a, b = torch.einsum("ka,eba...->keb...", self.end, G), torch.einsum("kb,eba...->kea...", self.end, G)
        return torch.stack([a[0], a[1], b[0], b[1]], 1)

    def diff(self, X, r):
        G = X.reshape(self.E, self.n, self.n, *X.shape[2:])
        return torch.einsum("ij,ebj...->ebi..." if r == 0 else "ij,eja...->eia...", self.D, G).reshape(X.shape)

    def lift(self, Hf, r):  # spread the two faces of axis r along it
        k = "ka,ekb...->eba..." if r == 0 else "kb,eka...->eba..."
        return torch.einsum(k, self.lift1, Hf[:, 2 * r:2 * r + 2]).reshape(self.E, self.n**2, *Hf.shape[3:])

    def residual(self, U, view):
        Uf = self.faces(U)
        Un = Uf[self.nbr, self.nbf]
        im = self.imp[:, None, None, None]
        ubar = torch.where(self.trace, view, torch.where(self.imex, torch.where(im, Un, Uf), 0.5 * (Uf + Un)))
        G = torch.stack([self.diff(U, r) + self.lift(ubar - Uf, r) for r in (0, 1)], 2)
        q = torch.einsum("esrc,esrv->escv", self.S, G) / self.J[..., None, None]
        qf = self.faces(q)
        qn = qf[self.nbr, self.nbf]
        Ft = torch.einsum("esrc,escv->esrv", self.S, self.conv(U) - self.visc(U, q))
        sg = torch.tensor([-1.0, 1.0, -1.0, 1.0], dtype=torch.float64, device=DEV)[:, None, None]
        Ftf = self.faces(Ft)
        own = sg * torch.cat([Ftf[:, :2, :, 0], Ftf[:, 2:, :, 1]], 1)
        dot = lambda F: torch.einsum("...cv,...c->...v", F, self.nrm)  # noqa: E731
        uh = torch.where(self.trace, view, Uf)
        hyb = dot(self.conv(uh) - self.visc(uh, qf)) + self.speed(uh, True)[..., None] * (Uf - uh)
        lam = torch.maximum(self.speed(Uf, False), self.speed(Un, False))[..., None]
        fr = 0.5 * dot(self.conv(Uf) + self.conv(Un)) + 0.5 * lam * (Uf - Un)
        vf, vn = dot(self.visc(Uf, qf)), dot(self.visc(Un, qn))
        fr = fr - torch.where(self.imex, torch.where(im, vf, vn), 0.5 * (vf + vn))
        Fn = self.Jf[..., None] * torch.where(self.trace, hyb, fr)
        # sigma g' on both ends: the lift above carries g' alone
        H = sg * (Fn - own)
        div = sum(self.diff(Ft[:, :, r], r) + self.lift(H, r) for r in (0, 1))
        return -div / self.J[..., None], torch.where(self.trace, self.w[:, None] * Fn, torch.zeros_like(Fn))

    def view(self, uhat):
        return torch.cat([uhat, torch.zeros_like(uhat[:1])])[self.tr]

    def gather(self, V):  # sum of the element faces' values on each trace
        out = torch.zeros(self.ntrace + 1, *V.shape[2:], dtype=V.dtype, device=DEV)
        return out.index_add_(0, self.tr.reshape(-1), V.reshape(-1, *V.shape[2:]))[:-1]

    def first_trace(self, U):
        return 0.5 * self.gather(torch.where(self.trace, self.faces(U), torch.zeros((), dtype=torch.float64, device=DEV)))

    def blocks(self, U, uhat, adt):
        """A, B, C, D of the implicit elements, one unknown of all elements together at a time."""
        v, k = self.view(uhat), self.imp.nonzero()[:, 0]
        nA, nT = self.n**2 * self.nv, 4 * self.n * self.nv

        def column(dU, dv):
            _, (dR, dg) = torch.func.jvp(self.residual, (U, v), (dU, dv))
            return torch.cat([(dU - adt * dR)[k].reshape(len(k), nA), dg[k].reshape(len(k), nT)], 1)

        cols, many = [], max(1, min(24, 20_000_000 // U.numel()))
        for j in range(0, nA + nT, many):
            d = torch.zeros(min(many, nA + nT - j), self.E, nA + nT, dtype=U.dtype, device=DEV)
            for i in range(len(d)):
                d[i, k, j + i] = 1.0
            cols.append(torch.func.vmap(column)(d[..., :nA].reshape(-1, *U.shape), d[..., nA:].reshape(-1, *v.shape)))
        M = torch.cat(cols).permute(1, 2, 0)
        return M[:, :nA, :nA], M[:, :nA, nA:], M[:, nA:, :nA], M[:, nA:, nA:]

    def precond(self, S):  # inverse of each trace's sum of diagonal face blocks
        bs = self.n * self.nv
        d = S.reshape(len(S), 4, bs, 4, bs)
        d = torch.stack([d[:, f, :, f] for f in range(4)], 1)
        P = torch.zeros(self.ntrace + 1, bs, bs, dtype=S.dtype, device=DEV)
        return torch.linalg.inv(P.index_add_(0, self.tr[self.imp].reshape(-1), d.reshape(-1, bs, bs))[:-1])

    def solve_trace(self, S, t, rtol=1e-9, m=60):
        """Right-preconditioned restarted GMRES on the assembled trace system."""
        bs, tr, P = self.n * self.nv, self.tr[self.imp], self.precond(S)
        add = lambda y: torch.zeros(self.ntrace + 1, bs, dtype=S.dtype, device=DEV).index_add_(0, tr.reshape(-1), y.reshape(-1, bs))[:-1]  # noqa: E731
        op = lambda x: add(torch.bmm(S, torch.cat([x, x[:1] * 0])[tr].reshape(len(S), -1, 1)))  # noqa: E731
        b, x = add(t), torch.zeros(self.ntrace, bs, dtype=S.dtype, device=DEV)
        if not self.ntrace:
            return x
        stop = rtol * float(b.norm())
        for _ in range(40):
            r = b - op(x)
            beta = float(r.norm())
            if beta <= stop:
                break
            V, H = [r / beta], np.zeros((m + 1, m))
            for j in range(m):
                w = op(torch.bmm(P, V[j][..., None])[..., 0])
                for _twice in (0, 1):
                    Q = torch.stack([q.reshape(-1) for q in V])
                    h = Q @ w.reshape(-1)
                    w = w - (h @ Q).reshape(w.shape)
                    H[:j + 1, j] += h.cpu().numpy()
                H[j + 1, j] = float(w.norm())
                e = np.zeros(j + 2)
                e[0] = beta
                y, res = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[:2]
                if j == m - 1 or (res.size and math.sqrt(max(res[0], 0.0)) <= stop) or H[j + 1, j] == 0.0:
                    break
                V.append(w / H[j + 1, j])
            z = sum(float(c) * q for c, q in zip(y, V))
            x = x + torch.bmm(P, z[..., None])[..., 0]
        return x

    def stage(self, U, uhat, Ustar, adt):
        """Newton on u - u* - adt R(u, u^) = 0, g = 0 to rounding."""
        k, first, last = self.imp.nonzero()[:, 0], None, math.inf
        for it in range(12):
            R, gv = self.residual(U, self.view(uhat))
            h, g = (U - Ustar - adt * R)[k], self.gather(gv)
            now = math.sqrt(float((h * h).sum() + (g * g).sum()))
            first = now if first is None else first
            if now <= 1e-13 * first or (it > 3 and now > 0.5 * last):
                break
            last = now
            A, B, C, D = self.blocks(U, uhat, adt)
            X = torch.linalg.solve(A, torch.cat([B, -h.reshape(len(k), -1, 1)], 2))
            S = D - C @ X[..., :-1]
            t = -gv[k].reshape(len(k), -1) - (C @ X[..., -1:])[..., 0]
            dh = self.solve_trace(S, t).reshape(uhat.shape)
            du = X[..., -1] - torch.bmm(X[..., :-1], self.view(dh)[k].reshape(len(k), -1, 1))[..., 0]
            U, uhat = U.clone(), uhat + dh
            U[k] += du.reshape(len(k), *U.shape[1:])
        return U, uhat, R

    def step(self, U, uhat, dt, tableau):
        if tableau == "be":
            a, b, ah, bh = [[1.0]], [1.0], [[], [1.0]], [0.0, 1.0]
        else:
            g, dl = 1 - 0.5**0.5, -2 * 2**0.5 / 3
            a, b, ah, bh = [[g], [1 - g, g]], [1 - g, g], [[], [g], [dl, 1 - dl]], [0.0, 1 - g, g]
        im = self.imp[:, None, None]
        Rs = [self.residual(U, self.view(uhat))[0]]
        for i in range(1, len(b) + 1):
            star = U + dt * sum((a[i - 1][j - 1] * Rs[j] for j in range(1, i)), torch.zeros_like(U))
            ex = U + dt * sum(ah[i][j] * Rs[j] for j in range(i))
            _, uhat, R = out = self.stage(torch.where(im, star, ex), uhat, star, a[i - 1][i - 1] * dt)
            Rs.append(R)
        del out
        return U + dt * torch.where(im, sum(c * R for c, R in zip(b, Rs[1:])), sum(c * R for c, R in zip(bh, Rs))), uhat

    def filter(self, U, alpha, s, eta_c):
        p = self.n - 1
        eta = np.add.outer(np.arange(self.n), np.arange(self.n))
        lam = np.where(eta < eta_c, 1.0, np.exp(-alpha * (np.maximum(eta - eta_c, 0) / (2 * p - eta_c)) ** s))
        V, Vi, lam = (torch.as_tensor(x, device=DEV) for x in (self.V, self.Vi, lam))
        G = U.reshape(self.E, self.n, self.n, self.nv)
        m = torch.einsum("bk,al,kl,kj,li,ejiv->ebav", V, V, lam, Vi, Vi, G)
        return m.reshape(U.shape)


def exact(case, seed):
    """The results of `run` in plain 64-bit torch; None where it would take too long (the largest mesh)
    or where the operator has no form here (mixed degree with walls, hexahedra, the embedded trace)."""
    if case["kind"] == "uneven":
        nA, nT, (A, B, C, D, r, s) = _uneven_problem(case, seed)
        sizes = list(zip(nA, nT))
        cut = lambda x, n: list(torch.split(x, n))  # noqa: E731
        A, B, C = cut(A, [a * a for a in nA]), cut(B, [a * t for a, t in sizes]), cut(C, [a * t for a, t in sizes])
        D, r, s = cut(D, [t * t for t in nT]), cut(r, nA), cut(s, nT)
        out = {k: [None] * len(nA) for k in ("XB", "xr", "S", "t")}
        for shape in sorted(set(sizes)):
            at, (a, t) = [i for i, z in enumerate(sizes) if z == shape], shape
            get = lambda x, *sh: torch.stack([x[i] for i in at]).view(len(at), *sh)  # noqa: E731
            X = torch.linalg.solve(get(A, a, a), torch.cat([get(B, a, t), get(r, a, 1)], 2))
            Y = get(C, t, a) @ X
            for k, v in (("XB", X[..., :-1]), ("xr", X[..., -1]), ("S", get(D, t, t) - Y[..., :-1]), ("t", get(s, t) - Y[..., -1])):
                for i, q in zip(at, v):
                    out[k][i] = q.reshape(-1)
        return {"LU": None, "piv": None, **{k: torch.cat(v) for k, v in out.items()}}
    if case["kind"] in ("wall", "channel", "efr") or case["nx"] * case["ny"] * (case["p"] + 1) ** 4 > 4_500_000:
        if case["kind"] != "residual":
            return None
    mesh, physics, u, dt = _periodic_problem(case, seed)
    op = Plain(mesh, physics)
    U = torch.as_tensor(u, dtype=torch.float64, device=DEV)
    uhat = op.first_trace(U)
    if case["kind"] == "residual":
        R, gv = op.residual(U, op.view(uhat))
        return R, op.gather(gv)
    g = 1 - 0.5**0.5
    if case["kind"] == "operator":
        A, B, C, D = op.blocks(U, uhat, g * dt)
        XB = torch.linalg.solve(A, B)
        S = D - C @ XB
        return {"S": S, "XB": XB, "Pinv": op.precond(S)}
    if case["kind"] == "stage":
        R0 = op.residual(U, op.view(uhat))[0]
        U1, uhat, R = op.stage(U, uhat, U, g * dt)
        return U1, uhat, torch.stack([R0, R])
    for _ in range(case["steps"]):
        U, uhat = op.step(U, uhat, dt, case["tableau"])
    if case["filter"]:
        U = op.filter(U, 36.0, 4.0, case["p"])
    return U, uhat
