"""(sigma, mu) of the eigenvalues that remedy R2 computes do not move with the arithmetic of the solves.

R2 shifts to sigma = fl(lambda) of an ill-conditioned first solve: its rounding, K_nu times larger than
that of lambda, is the returned sigma.  The solve of such an eigenvalue therefore has one fixed arithmetic
(condition above 2^20), and the others may move by at most 2^20 roundings of their terms, 8 ulps or so.
"""
import os

import numpy as np
import pytest
import torch

from paper_1405_7537_gb300 import binding, workloads as W
from gpu_common import two_sum

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "r2_shifts.txt")


def _records():
    out = []
    for line in open(GOLDEN):
        if line.startswith("#"):
            continue
        f = line.split()
        if f[0] in ("eig", "arrow"):
            out.append((tuple(f), []))
        else:
            out[-1][1].append((int(f[0]), float.fromhex(f[1]), float.fromhex(f[2])))
    return out


def _clustered(seed):
    rng = np.random.default_rng(seed)
    c = rng.uniform(-1, 1, 40)
    d = np.sort(rng.choice(c, 240) + rng.choice([1.0, -1.0], 240) * 10.0 ** rng.uniform(-12, -3, 240))[::-1].copy()
    return d, rng.choice([1.0, -1.0], 240) * 10.0 ** rng.uniform(-12, 0, 240), 1e-5


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs CUDA")
    return binding


@pytest.mark.parametrize("rec", _records(), ids=lambda r: "-".join(r[0]))
def test_shift_of_an_ill_conditioned_eigenvalue(B, rec):
    (kind, spectrum, n, seed, finder), pairs = rec
    n, seed = int(n), int(seed)
    if spectrum == "clustered":
        d, z, par = _clustered(seed)
    elif kind == "arrow":
        d, z, par = W.arrowhead(n, seed)
    else:
        d, z, par = W.large(n, seed, with_W=False)[:3] if spectrum == "large" else getattr(W, spectrum)(n, seed)
    solve = B.eig if kind == "eig" else B.eig_arrowhead
    r = solve(torch.tensor(d, device="cuda"), torch.tensor(z, device="cuda"), float(par), want_vectors=False,
              options=B.default_options(zero_finder=int(finder)), check=True)
    s, m = r["sigma"].cpu().numpy(), r["mu"].cpu().numpy()
    k, s0, m0 = (np.array(c) for c in zip(*pairs))
    gap = np.min(np.abs(s0[:, None] - d[None, :]), axis=1)
    assert np.all(np.abs(s[k] - s0) <= 2.0 ** -30 * gap + 2 * np.spacing(np.abs(s0)))
    # and the same lambda = sigma + mu to the accuracy of mu
    x, e = two_sum(s[k], -s0)
    assert np.all(np.abs(x + (e + (m[k] - m0))) <= 64 * 2.0 ** -52 * (np.abs(m[k]) + np.abs(m0) + np.abs(x)))
