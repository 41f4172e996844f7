"""The scalar operations against extended precision: mantissas drawn at random and at the edges of the
reciprocal's seed (next to 1 and 2, next to and on the 24-bit numbers), over the whole exponent range."""
import numpy as np
import pytest
import torch

from paper_1405_7537_gb300 import binding

pytestmark = pytest.mark.gpu
RCP, RCP_EVAL, QUOT, QUOT_ROUGH, ROOT, MAG = range(6)


def numbers(lo, hi, seed, count=1 << 18):
    """Signed binary64 numbers with exponents from lo to hi."""
    rng = np.random.default_rng(seed)
    k = rng.integers(0, 1 << 20, 4096)
    grid = rng.integers(1 << 23, 1 << 24, 4096) << 29                            # 24-bit mantissas
    edge = np.concatenate([(1 << 52) + k, (1 << 53) - 1 - k, grid, grid + 1, grid - 1, grid + (1 << 29) - 1,
                           grid + (1 << 28), (1 << 52) + np.arange(64), (1 << 53) - 1 - np.arange(64)])
    m = np.concatenate([edge.clip(1 << 52, (1 << 53) - 1), rng.integers(1 << 52, 1 << 53, count)])
    return np.ldexp(m.astype(np.float64), rng.integers(lo, hi + 1, m.size) - 52) * rng.choice([-1.0, 1.0], m.size)


def run(which, a, b=None):
    if not torch.cuda.is_available():
        pytest.skip("needs CUDA")
    t = lambda x: None if x is None else torch.tensor(x, device="cuda")          # noqa: E731
    return binding.probe_scalar(which, t(a), t(b)).cpu().numpy()


def ulps(r, exact):
    return (np.abs(r.astype(np.longdouble) - exact) / np.spacing(np.abs(exact.astype(np.float64)))).astype(np.float64)


# the last Newton step leaves half an ulp of rounding and the square of the seed's error: 2^-90 for the
# seed within 2^-45, the cube 2^-57 of the 19-bit seed (2^-4 ulp)
@pytest.mark.parametrize("which,bound", [(RCP, 0.51), (RCP_EVAL, 0.57)])
def test_reciprocals(which, bound):
    x = numbers(-1020, 1019, 1)
    assert ulps(run(which, x), 1 / x.astype(np.longdouble)).max() <= bound
    out = np.array([2.0 ** 1023, 1.5 * 2.0 ** 1023, 2.0 ** -1022, 2.0 ** -1021, np.inf, -np.inf])
    assert np.array_equal(run(which, out), 1 / out)                               # the IEEE quotient out of range


def test_quotients():
    a, b = numbers(-400, 400, 2), numbers(-500, 500, 3)
    exact = a.astype(np.longdouble) / b.astype(np.longdouble)
    assert ulps(run(QUOT, a, b), exact).max() <= 2.0
    rel = np.abs(run(QUOT_ROUGH, a, b).astype(np.longdouble) / exact - 1)
    assert rel.max() <= 2.0 ** -38


def test_square_root():
    x = np.abs(numbers(-1021, 1023, 4))
    assert ulps(run(ROOT, x), np.sqrt(x.astype(np.longdouble))).max() <= 2.0
    s = np.array([0.0, np.inf, 2.0 ** -1074, 2.0 ** -968, 2.0 ** 967])
    assert np.array_equal(run(ROOT, s), np.sqrt(s))


def test_truncated_magnitude():
    x = numbers(-126, 127, 5)
    r = run(MAG, x)
    assert np.array_equal(r, r.astype(np.float32)) and np.all(r <= np.abs(x)) and np.all(r > np.abs(x) * (1 - 2.0 ** -23))
