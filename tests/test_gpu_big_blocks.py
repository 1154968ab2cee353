"""Condensation of blocks too large for one CTA's shared memory (the blocked LU, the column-block
solve, the Schur product) at the edges of its tiles: panels of 32 / 16 pivots, column blocks of 16 to
128, product tiles of 128 and 256, block sides that are no multiple of a 16-byte vector, and the
variants' row limits, each with its rows shuffled so that every panel interchanges.

Tolerances: FP64 1e-11 relative to the largest value (condition numbers of a few units).  FP32:
nA 2^-24 bounds the accumulated rounding of an nA-term substitution, and 2e-5 covers the 3xTF32
products of S (2^-21 per term) at the smaller sizes."""

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

FP32 = [[(65, 1)], [(67, 62), (96, 63)], [(97, 64), (100, 96)], [(128, 127), (129, 128), (144, 129)], [(135, 270)],
        [(256, 255), (90, 40)], [(320, 257)], [(341, 130)], [(400, 33)], [(700, 20)]]
FP64 = [[(129, 1)], [(130, 15), (144, 16)], [(145, 63), (144, 64)], [(135, 270)], [(200, 31)], [(320, 33)], [(400, 17)],
        [(800, 5)]]


@pytest.mark.parametrize("prec,shapes", [(p, s) for p, g in (("fp32", FP32), ("fp64", FP64)) for s in g])
def test_large_blocks_at_tile_edges(prec, shapes):
    rng = np.random.default_rng(3)
    shapes = shapes * 2
    blocks = []
    for nA, nT in shapes:
        A = 4.0 * np.eye(nA) + rng.standard_normal((nA, nA)) / np.sqrt(nA)
        blocks.append((A[rng.permutation(nA)], rng.standard_normal((nA, nT)), rng.standard_normal((nT, nA)),
                       rng.standard_normal((nT, nT)), rng.standard_normal(nA), rng.standard_normal(nT)))
    dtype = torch.float64 if prec == "fp64" else torch.float32
    packed = [torch.tensor(np.concatenate([b[i].reshape(-1) for b in blocks]), dtype=dtype if i < 4 else torch.float64,
                           device="cuda") for i in range(6)]
    out = pkg.hfr_condense_uneven([a for a, _ in shapes], [t for _, t in shapes], *packed,
                                  precision=pkg.FR_PREC_FP64 if prec == "fp64" else pkg.FR_PREC_FP32)
    got = {k: out[k].cpu().numpy().astype(np.float64) for k in ("XB", "xr", "S", "t")}
    o = dict.fromkeys(got, 0)
    for k, (b, (nA, nT)) in enumerate(zip(blocks, shapes)):
        if prec == "fp32":  # the oracle on the rounded blocks
            b = tuple(x.astype(np.float32).astype(np.float64) if i < 4 else x for i, x in enumerate(b))
        tol = 1e-11 if prec == "fp64" else max(2e-5, nA * 2.0**-24)
        for name, ref in zip(("XB", "xr", "S", "t"), condense(*(x[None] for x in b))):
            ref = ref[0].reshape(-1)
            err = np.abs(got[name][o[name]:o[name] + ref.size] - ref).max() / np.abs(ref).max()
            assert err < tol, (name, k, (nA, nT), err)
            o[name] += ref.size
