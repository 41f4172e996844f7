"""The adjoint is linear in the cotangents, also where they are tiny and a row's components are (a
rank-one part far above the poles: x_j = z_j / (d_j - lambda) of the exterior eigenvalue)."""
import numpy as np
import pytest

from test_gpu_backward import B, cu  # noqa: F401
from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho,shift", [(1e40, 700), (1e60, 700), (1e65, 600), (1.0, 700)])
@pytest.mark.parametrize("n", [33, 300])
def test_tiny_cotangents(B, rho, shift, n):  # noqa: F811
    """Scaling by a power of two commutes with every rounding; grad_rho at rho >> 1 is the exterior row's."""
    d, z, _ = W.uniform(n, 3)
    r = B.eig(cu(d), cu(z), rho)
    rng = np.random.default_rng(n)
    w, Wm = rng.standard_normal(n), rng.standard_normal((n, n))
    a = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], None, cu(Wm))
    b = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], None, cu(np.ldexp(Wm, -shift)))
    for x, y in zip(a, b):
        x, y = x.cpu().numpy(), np.ldexp(y.cpu().numpy(), shift)
        assert np.all(np.abs(x - y) <= 1e-12 * np.max(np.abs(x)))
    c = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], cu(np.ldexp(w, -shift)), cu(np.ldexp(Wm, -shift)))
    e = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], cu(w), cu(Wm))
    for x, y in zip(e, c):
        x, y = x.cpu().numpy(), np.ldexp(y.cpu().numpy(), shift)
        assert np.all(np.abs(x - y) <= 1e-12 * np.max(np.abs(x)))
