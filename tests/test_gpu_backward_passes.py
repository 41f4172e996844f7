"""The adjoint's row kernel holds each lane's largest component out of its sums while it looks for the
row's largest: orders around the lane width and the warp counts' limits, rows whose components tie or are
dominated by one entry, data far outside the range of its plain sums (they are formed again in units of
v), either cotangent alone, a workspace of the fewer partial rows, against the oracle's adjoint component
by component (the bound of test_gpu_backward)."""
import numpy as np
import pytest

import oracle
from adjoint_scale import adjoint_scales
from test_gpu_backward import B, check_components, cu  # noqa: F401
from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(kind, n):
    d, z, rho = W.uniform(n, n)
    if kind == "ties":                               # mirrored poles: pairs of equal components
        d = np.concatenate([np.linspace(1, 0.1, n - n // 2), -np.linspace(0.1, 1, n // 2)])
        z = np.ones(n)
    elif kind == "dominated":                        # eigenvectors within 1e-10 of a unit vector
        z = z * 1e-6
    elif kind == "far":                              # x up to 1e130: sums of squares leave the range
        rho = 1e-140
    return d, z, rho


@pytest.mark.parametrize("kind", ["uniform", "ties", "dominated", "far"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 65, 1065])
@pytest.mark.parametrize("parts", ["both", "lambda", "V"])
def test_against_oracle(B, kind, n, parts):  # noqa: F811
    if n == 1 and parts == "V":
        pytest.skip("V = [1]: every gradient is exactly zero, with no scale to compare at")
    d, z, rho = _problem(kind, n)
    rng = np.random.default_rng(n)
    w = rng.standard_normal(n) if parts != "V" else None
    Wm = rng.standard_normal((n, n)) if parts != "lambda" else None
    r = B.eig(cu(d), cu(z), rho)
    gd, gz, gr = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], cu(w) if w is not None else None,
                                cu(Wm) if Wm is not None else None)
    sig, mu = r["sigma"].cpu().numpy(), r["mu"].cpu().numpy()
    w0, W0 = (w if w is not None else np.zeros(n)), (Wm if Wm is not None else np.zeros((n, n)))
    ref = oracle.backward(d, z, rho, sig, mu, w0, W0)
    check_components((gd.cpu().numpy(), gz.cpu().numpy(), gr.item()), ref,
                     adjoint_scales(d, z, rho, sig, mu, w0, W0), n, (kind, n, parts))


def test_smaller_workspace(B):  # noqa: F811
    n = 3100
    d, z, rho = W.uniform(n, 5)
    r = B.eig(cu(d), cu(z), rho, want_vectors=False)
    w = torch.randn(n, dtype=torch.float64, device="cuda")
    size = int(B.lib().dpr1_backward_workspace_size(n))
    full = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], w)
    part = torch.empty(size // 2 + 100000, dtype=torch.uint8, device="cuda")
    less = B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], w, ws=part)
    for a, b in zip(full, less):
        assert torch.allclose(a, b, rtol=1e-10, atol=1e-10 * float(a.abs().max()))
    with pytest.raises(B.DPR1Error):
        B.eig_backward(cu(d), cu(z), rho, r["sigma"], r["mu"], w, ws=part[:size // 2 - 200000])


def test_not_a_number_is_reported(B):  # noqa: F811
    n = 70
    d, z, rho = W.uniform(n, 6)
    r = B.eig(cu(d), cu(z), rho)
    G = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    G[3, 64] = float("nan")
    z2 = cu(z)
    z2[5] = 0.0                                      # 0 / 0 at the pole of a deflated weight
    sig, mu = r["sigma"].clone(), r["mu"].clone()
    mu[7] = 0.0
    for args in ((cu(z), r["sigma"], r["mu"], G), (z2, sig, mu, torch.zeros_like(G))):
        with pytest.raises(B.DPR1Error) as e:
            B.eig_backward(cu(d), args[0], rho, args[1], args[2], None, args[3])
        assert e.value.code == 4
