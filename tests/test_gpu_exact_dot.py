"""Reproducible dot at the edges of its kernel: lengths around a block's and a
launch's step, and products around a thread's window (placed by the block's
first ones): later ones above it and below it, subnormals, infinities and NaN.
Bit for bit the oracle's correctly rounded sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STEP = 512 * 4


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2311_13914_gb300 import _build, binding

    _build.build()
    return binding


def _same(a, b):
    return np.float64(a).view(np.uint64) == np.float64(b).view(np.uint64) or (np.isnan(a) and np.isnan(b))


@pytest.mark.parametrize("n", [1, 31, 512, STEP - 1, STEP + 1, 304 * STEP - 1, 304 * STEP + 1, 2 * 304 * STEP + 7])
def test_lengths(B, oracle_lib, n):
    import torch

    rng = np.random.default_rng(n)
    x, y = rng.standard_normal(n), rng.standard_normal(n)
    want = oracle_lib.dot_exact(x, y)
    xd, yd = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
    assert _same(B.bd_dot_exact(xd, yd), want)
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert _same(B.bd_dot_exact_noalloc(xd, yd, out).item(), want)
    if n > 1:  # 8-byte aligned starts
        assert _same(B.bd_dot_exact(xd[1:], yd[1:]), oracle_lib.dot_exact(x[1:], y[1:]))


@pytest.mark.parametrize("first,later", [(0, 9), (0, 10), (0, 400), (0, -127), (0, -128), (0, -161), (0, -900),
                                         (-1000, 0), (-537, -537), (-537, -530), (511, 511), (511, -500)])
def test_windows(B, oracle_lib, first, later):
    """Magnitudes 2^(2 first) in the block's first products, 2^(2 later) after."""
    rng = np.random.default_rng(abs(first) + abs(later))
    n = 5 * STEP + 3
    e = np.where(np.arange(n) < 2 * STEP, first, later)
    x, y = np.ldexp(rng.standard_normal(n), e), np.ldexp(rng.standard_normal(n), e)
    assert _same(B.bd_dot_exact(x, y), oracle_lib.dot_exact(x, y))
    z = np.concatenate([x, -x[::-1], [2.0 ** -600]])  # everything cancels but the last product
    w = np.concatenate([y, y[::-1], [1.0]])
    assert _same(B.bd_dot_exact(z, w), oracle_lib.dot_exact(z, w))


def test_special_values(B):
    x = np.ones(3 * STEP)
    for at, want in (({5: np.inf}, np.inf), ({5: -np.inf}, -np.inf), ({5: np.inf, 4000: -np.inf}, np.nan),
                     ({6000: np.nan}, np.nan)):
        y = np.ones(3 * STEP)
        for i, v in at.items():
            y[i] = v
        assert _same(B.bd_dot_exact(x, y), want)
