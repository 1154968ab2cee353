"""Condensation of blocks that fill a CTA's shared memory to the last bytes (227 KB): FP64 blocks of the
LU kernel and of the shared-memory Gauss-Jordan elimination, FP32 blocks of the latter, through the
allocation-free call and the uneven batch; and the shapes just beyond, which other kernels take.

Tolerances: diagonally dominant blocks with condition numbers below 100 and rows up to 4842 long: FP64
1e-11, FP32 1e-4 of the largest value."""

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
from oracle.solve import condense  # noqa: E402

LU64 = [(128, 96), (128, 97), (128, 98), (149, 44), (149, 45), (64, 226), (65, 223), (160, 20), (13, 1117), (127, 99),
        (127, 100)]
GJ64 = [(112, 31), (112, 32), (109, 44), (89, 116), (119, 2), (42, 319), (37, 367)]
GJ32 = [(52, 525), (43, 644), (40, 695), (40, 696)]


def blocks(rng, nA, nT, n):
    A = 4.0 * np.eye(nA) + rng.standard_normal((n, nA, nA)) / np.sqrt(nA)
    A = A[:, rng.permutation(nA)]
    return (A, rng.standard_normal((n, nA, nT)), rng.standard_normal((n, nT, nA)) / np.sqrt(nA),
            rng.standard_normal((n, nT, nT)), rng.standard_normal((n, nA)), rng.standard_normal((n, nT)))


def check(got, b, tol):
    for name, g, ref in zip(("XB", "xr", "S", "t"), got, condense(*b)):
        err = np.abs(g.reshape(ref.shape) - ref).max() / np.abs(ref).max()
        assert err < tol, (name, err)


@pytest.mark.parametrize("nA,nT", LU64 + GJ64)
def test_uniform_fp64(nA, nT):
    n = 3
    b = blocks(np.random.default_rng(nA + nT), nA, nT, n)
    A, B, C, D, r, s = (torch.tensor(x, device="cuda").contiguous() for x in b)
    XB, S, xr, t = torch.empty_like(B), torch.empty_like(D), torch.empty_like(r), torch.empty_like(s)
    assert pkg.hfr_condense_noalloc(A, B, C, D, r, s, XB, xr, S, t, precision=pkg.FR_PREC_FP64) == 0
    check([x.cpu().numpy() for x in (XB, xr, S, t)], b, 1e-11)


@pytest.mark.parametrize("prec,nA,nT", [("fp64", *x) for x in GJ64] + [("fp32", *x) for x in GJ32])
def test_uneven_batch(prec, nA, nT):
    """the filling shape among smaller ones, whose bundles share its launch"""
    rng = np.random.default_rng(nA * nT)
    shapes = [(nA, nT), (9, 12), (16, 16), (nA, nT), (9, 12)]
    bl = [blocks(rng, a, t, 1) for a, t in shapes]
    dt = torch.float64 if prec == "fp64" else torch.float32
    packed = [torch.tensor(np.concatenate([b[i].reshape(-1) for b in bl]), dtype=dt if i < 4 else torch.float64,
                           device="cuda") for i in range(6)]
    out = pkg.hfr_condense_uneven([a for a, _ in shapes], [t for _, t in shapes], *packed,
                                  precision=pkg.FR_PREC_FP64 if prec == "fp64" else pkg.FR_PREC_FP32)
    got = [out[k].cpu().numpy().astype(np.float64) for k in ("XB", "xr", "S", "t")]
    o = [0, 0, 0, 0]
    for b, (a, t) in zip(bl, shapes):
        if prec == "fp32":
            b = tuple(x.astype(np.float32).astype(np.float64) if i < 4 else x for i, x in enumerate(b))
        size = (a * t, a, t * t, t)
        check([g[p:p + m] for g, p, m in zip(got, o, size)], b, 1e-11 if prec == "fp64" else 1e-4)
        o = [p + m for p, m in zip(o, size)]
