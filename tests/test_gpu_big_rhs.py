"""x_r and t of FP32 batches with a block of more than 894 rows: the right-hand side keeps its 64 bits
through the substitution, in every large block of the batch.

The blocks' factors are exact in FP32: A = P^T L U with L unit lower and U upper bidiagonal, entries
dyadic, |l| <= 1/2 (so that partial pivoting finds the rows of L U again) and each intermediate value a
sum of two short dyadic numbers.  The only rounding of x_r is then the FP64 substitution's: with
||A^-1|| ||A|| below 100, a few units of 2^-53 times 100 stay under 1e-12; t adds nA products, 1e-12
relative to the largest |c_ij x_j| sum.  A right-hand side rounded to FP32 is off by 3e-8."""

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


def exact_block(rng, nA):
    Lo = np.eye(nA) + np.diag(rng.choice([-0.5, -0.25, 0.25, 0.5], nA - 1), -1)
    U = np.diag(rng.choice([-4.0, -2.0, 2.0, 4.0], nA)) + np.diag(rng.choice([-0.5, 0.0, 0.5], nA - 1), 1)
    return (Lo @ U)[rng.permutation(nA)]


@pytest.mark.parametrize("shapes", [[(895, 3)], [(900, 33), (130, 40)], [(1023, 2)], [(70, 5), (1024, 17)]])
def test_right_hand_side_keeps_64_bits(shapes):
    rng = np.random.default_rng(5)
    blocks = [(exact_block(rng, nA), rng.standard_normal((nA, nT)), rng.integers(-8, 9, (nT, nA)) / 4.0,
               rng.standard_normal((nT, nT)), rng.standard_normal(nA), rng.standard_normal(nT)) for nA, nT in shapes]
    packed = [torch.tensor(np.concatenate([b[i].reshape(-1) for b in blocks]),
                           dtype=torch.float32 if i < 4 else torch.float64, device="cuda") for i in range(6)]
    out = pkg.hfr_condense_uneven([a for a, _ in shapes], [t for _, t in shapes], *packed, precision=pkg.FR_PREC_FP32)
    xr, t = out["xr"].cpu().numpy(), out["t"].cpu().numpy()
    oa = ot = 0
    for (nA, nT), (A, _, C, _, r, s) in zip(shapes, blocks):
        ref = np.linalg.solve(A, r)
        assert np.abs(xr[oa:oa + nA] - ref).max() < 1e-12 * np.abs(ref).max(), (nA, nT)
        assert np.abs(t[ot:ot + nT] - (s - C @ ref)).max() < 1e-12 * (np.abs(C) @ np.abs(ref)).max(), (nA, nT)
        oa += nA
        ot += nT
