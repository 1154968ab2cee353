"""The quotients of the column-block solve: with diagonal blocks A = diag(d) the entries of X = A^{-1} B
are single quotients b / d, formed from the stored reciprocal and one correction.  Against exact
rational arithmetic over random operands and at the ends of the range (subnormal and largest
numerators, divisors and results, zeros, an overflow).

Tolerance: half a unit in the last place plus 2^-7 of one (2^-8 at the smallest numerator that is not
divided, and a few 2^-24 or 2^-53); a division itself stays within half a unit."""

from fractions import Fraction

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


def draw(rng, f, shape, e0, e1):
    """signed values of the type with exponents e0 .. e1 (subnormals where below its range)"""
    m = 1.0 + rng.random(shape)
    x = np.ldexp(m, rng.integers(e0, e1 + 1, shape)).astype(f)
    return np.where(rng.random(shape) < 0.5, -x, x).astype(f)


@pytest.mark.parametrize("f,nA,nT", [(np.float32, 128, 192), (np.float32, 320, 65), (np.float64, 144, 96)])
@pytest.mark.parametrize("span", ["ordinary", "tiny", "huge", "full"])
def test_quotients(f, nA, nT, span):
    rng = np.random.default_rng(nA + nT + len(span))
    lo, hi, sub = (-126, 126, -149) if f == np.float32 else (-1022, 1022, -1074)
    de, be = {"ordinary": ((-20, 20), (-20, 20)), "tiny": ((-3, 3), (sub, lo + 12)), "huge": ((hi - 2, hi), (hi - 9, hi)),
              "full": ((lo + 1, hi), (sub, hi))}[span]
    d = draw(rng, f, nA, *de)
    b = draw(rng, f, (nA, nT), *be)
    b[rng.random((nA, nT)) < 0.05] = 0.0
    with np.errstate(all="ignore"):
        q = b / d[:, None]
        b = np.where(np.isfinite(q), b, f(1.0) * d[:, None])  # an infinity would spread to the rows above
        if span == "full":  # but for the first row, which has none
            b[0, 3], d[0] = np.finfo(f).max, f(0.25)
        q = b / d[:, None]
    dt = torch.float32 if f == np.float32 else torch.float64
    dev = lambda x, t=dt: torch.tensor(np.ascontiguousarray(x).reshape(-1), dtype=t, device="cuda")
    out = pkg.hfr_condense_uneven([nA], [nT], dev(np.diag(d)), dev(b), dev(np.zeros((nT, nA), f)),
                                  dev(np.zeros((nT, nT), f)), dev(np.zeros(nA), torch.float64),
                                  dev(np.zeros(nT), torch.float64),
                                  precision=pkg.FR_PREC_FP32 if f == np.float32 else pkg.FR_PREC_FP64)
    x = out["XB"].cpu().numpy().reshape(nA, nT)
    assert np.array_equal(np.isfinite(x), np.isfinite(q)) and np.array_equal(x[~np.isfinite(x)], q[~np.isfinite(q)])
    off = np.argwhere((x != q) & np.isfinite(q))  # the division is correctly rounded: only these need a look
    assert len(off) <= 0.01 * x.size
    for i, j in off:
        exact = Fraction(float(b[i, j])) / Fraction(float(d[i]))
        ulp = Fraction(float(np.spacing(np.abs(q[i, j]))))
        assert abs(Fraction(float(x[i, j])) - exact) <= ulp * (Fraction(1, 2) + Fraction(1, 128)), (b[i, j], d[i], x[i, j])
