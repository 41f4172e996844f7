"""The products of the divide and conquer run over the rows and positions that do not deflate, and
deflated rows are copies: orders at the edges of the lists' chunks (1024) and of the product's
tiles (64), with nothing, something and everything deflated, ties and zero couplings among them.
Residual, orthogonality and LAPACK's eigenvalues as in test_gpu_tridiag (16 n u); the eigenvalues
are the same bits with and without eigenvectors (the columns kept without them are summed in the
products' order)."""
import numpy as np
import pytest

from test_gpu_tridiag import B, cu, props_gpu  # noqa: F401
from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "random":                            # most of every merge deflates
        return W.tridiagonal(n, n)
    if kind == "smooth":                            # hardly anything does
        return 2.0 + 1e-3 * np.cos(np.linspace(0, 3, n)), -np.ones(n - 1)
    if kind == "weak":                              # every coupling below the deflation tolerance
        return rng.uniform(-1, 1, n), np.full(n - 1, 1e-18)
    if kind == "uncoupled":                         # rho = 0 at every merge, ties in the poles
        return np.arange(float(n)) % 7, np.zeros(n - 1)
    b = np.ones(n - 1)                              # equal blocks of ten: ties with non-zero weights
    b[9::10] = np.where(np.arange(b[9::10].size) % 2 == 0, 0.0, 1e-9)
    return np.ones(n), b


@pytest.mark.parametrize("n", [63, 65, 129, 1025, 2049])
@pytest.mark.parametrize("kind", ["random", "smooth", "weak", "uncoupled", "blocks"])
def test_lists(B, kind, n):  # noqa: F811
    a, b = _matrix(kind, n)
    lam, Qt = B.eigh_tridiagonal(cu(a), cu(b))
    lam0, none = B.eigh_tridiagonal(cu(a), cu(b), want_vectors=False)
    assert none is None and torch.equal(lam, lam0)
    props_gpu(B, a, b, lam.cpu().numpy(), Qt.cpu().numpy())
