"""The recompute of eigenvalues much nearer to zero than to their poles (D + rho z z^T): by a warp in
problems of mean order up to 200, by a block above, from stored elements in every lane group."""
import numpy as np
import pytest
import torch

from paper_1405_7537_gb300 import binding
from gpu_common import tol

pytestmark = pytest.mark.gpu
cu = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")              # noqa: E731


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs CUDA")
    return binding


def problem(n, seed):
    """(d, z, rho, index, lambda): f(0) = 1 + rho sum z^2/d = 1e-4, so one eigenvalue next to zero, found by
    Newton's method in extended precision."""
    rng = np.random.default_rng(seed)
    d = np.sort(np.concatenate([rng.uniform(0.5, 1.0, n // 3), rng.uniform(-1.0, -0.25, n - n // 3)]))[::-1].copy()
    z = rng.uniform(0.5, 1.0, n) * rng.choice([1.0, -1.0], n)
    dl, zl = d.astype(np.longdouble), z.astype(np.longdouble)
    rho = float(-(1 - np.longdouble(1e-4)) / np.sum(zl * zl / dl))
    assert rho > 0
    lam, r = np.longdouble(0), np.longdouble(rho)
    for _ in range(6):
        x = dl - lam
        lam -= (1 + r * np.sum(zl * zl / x)) / (r * np.sum(zl * zl / (x * x)))
    return d, z, rho, n // 3, float(lam)


@pytest.mark.parametrize("n", [60, 200, 201, 700, 2500])
@pytest.mark.parametrize("finder", [0, 1])
def test_near_zero_eigenvalue(B, n, finder):
    d, z, rho, k, lam = problem(n, n)
    ws = B.workspace(n, "cuda")
    r = B.eig(cu(d), cu(z), rho, options=B.default_options(zero_finder=finder), ws=ws, check=True)
    assert B.workspace_stats(ws)["zero_path"] == 1
    # f(0) is 1e-4, its terms 1: 2^-63 of them (the extended precision) is 1e-15 of lambda
    assert abs(r["lam"][k].item() - lam) <= (tol(n) + 1e-15) * abs(lam)


@pytest.mark.parametrize("n", [20, 210])
def test_batch_of_more_candidates_than_buffers(B, n):
    """400 problems, a candidate each.  The recompute does not depend on the launch shape of the solve
    kernel, whose narrowest has fewer buffers than 400, nor on which lane group takes a candidate."""
    probs = [problem(n, s) for s in range(400)]
    sizes = [n] * len(probs)
    d, z = np.concatenate([p[0] for p in probs]), np.concatenate([p[1] for p in probs])
    rho = np.array([p[2] for p in probs])
    at = np.array([p * n + q[3] for p, q in enumerate(probs)])
    want = np.array([q[4] for q in probs])
    bt = B.Batch(sizes)
    res = []
    for opt in ({}, {"lanes": 32, "warps_per_block": 1, "blocks_per_sm": 1}):
        for _ in range(2):
            bt.solve(cu(d), cu(z), cu(rho), options=B.default_options(**opt), check=True)
            assert B.workspace_stats(bt.ws)["zero_path"] == len(probs)
            res.append(bt.lam.cpu().numpy()[at])
    assert np.all(np.abs(res[0] - want) <= (tol(n) + 1e-15) * np.abs(want))
    for r in res[1:]:
        assert np.array_equal(r.view(np.int64), res[0].view(np.int64))
