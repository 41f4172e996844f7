"""Eigenvector rows of a batch by 8, 16 or 32 lanes (mean order up to 128, up to 512, above): orders
around the lane widths and odd ones (rows that start off a 16-byte boundary), a problem that deflates
and one with rho = 0 among them, against single calls within 16 n 2^-53."""
import numpy as np
import pytest

from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1, 2, 7, 8, 9, 15, 17, 33, 100], [1, 129, 130, 257, 300, 511], [3, 700, 901]])
def test_rows_of_a_batch(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7537_gb300 import binding as B
    probs = [list(W.uniform(n, n)) for n in sizes]
    probs[-1][0] = probs[-1][0].copy()
    probs[-1][0][5] = probs[-1][0][4]                # a tie
    probs[-1][1] = probs[-1][1].copy()
    probs[-1][1][9] = 0.0                            # a zero weight
    probs[0][2] = 0.0
    cu = lambda x: torch.tensor(np.array(x, copy=True, order="C") + 0.0, device="cuda")  # noqa: E731
    b = B.Batch(sizes)
    b.Vt.fill_(float("nan"))
    b.solve(cu(np.concatenate([p[0] for p in probs])), cu(np.concatenate([p[1] for p in probs])),
            cu(np.array([p[2] for p in probs])), check=True)
    for i, (d, z, rho) in enumerate(probs):
        one = B.eig(cu(d), cu(z), rho)
        lam, Vt = b.block(i)
        tol = 16 * d.size * 2.0 ** -53
        assert ((lam - one["lam"]).abs() <= tol * one["lam"].abs()).all(), sizes[i]
        assert ((Vt - one["Vt"]).abs() <= tol * one["Vt"].abs()).all(), sizes[i]
