"""A batch that holds one problem of an order above 2048 takes the solve kernel's large form, whose idle
lane groups write eigenvector rows: the results are the single call's within the bound.  Orders on both
sides of the form's limit, and a block of eigenvectors that does not start at the array's beginning."""
import numpy as np
import pytest

from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(2048, 0), (2049, 0), (3000, 0), (3000, 6)])
def test_batch_of_one(n, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7537_gb300 import binding as B
    d, z, rho = W.uniform(n, n)
    dt, zt = torch.tensor(d, device="cuda"), torch.tensor(z, device="cuda")
    one = B.eig(dt, zt, rho)
    b = B.Batch([n])
    if shift:
        b.Vt = torch.empty(n * n + shift, dtype=torch.float64, device="cuda")
        b.voffs += shift
    b.Vt.fill_(float("nan"))
    b.solve(dt, zt, torch.tensor([rho], dtype=torch.float64, device="cuda"), check=True)
    # the two launches may differ in shape, and with it in the order of the sums
    tol = 16 * n * 2.0 ** -53
    V = b.Vt[shift:].view(n, n)
    assert torch.isfinite(V).all()
    assert ((b.lam - one["lam"]).abs() <= tol * one["lam"].abs()).all()
    assert ((V - one["Vt"]).abs() <= tol * one["Vt"].abs()).all()
