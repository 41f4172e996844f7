"""The finishing step of the solves (one evaluation with its slope in a bracket of 2^16 doubles in
place of the bisection's last steps): orders around the lane widths, the chunks of the evaluation
loop and the two compiled forms, both zero finders and every lane width, against the oracle within
16 n 2^-53; the exterior eigenvalues of a large rank-one part (declined: K_nu is large) and poles next
to the root (the evaluation repeated) among them.  On O(1) weights it leaves about one binary64
evaluation per eigenvalue (bounded by 3 here; 7 to 10 without it)."""
import numpy as np
import pytest

import oracle
from paper_1405_7537_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lanes", [(2, 0), (9, 8), (33, 32), (97, 0), (129, 8), (129, 32), (385, 0), (385, 16),
                                     (2047, 0), (2049, 0)])
@pytest.mark.parametrize("kind,finder", [("uniform", 0), ("uniform", 1), ("strong", 0), ("close", 0)])
def test_against_oracle(n, lanes, kind, finder):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7537_gb300 import binding as B
    d, z, rho = W.uniform(n, n)
    if kind == "strong":
        rho = 1e6
    elif kind == "close":
        z = z * 10.0 ** np.random.default_rng(n).uniform(-9, 0, n)
    ws = B.workspace(n)
    r = B.eig(torch.tensor(d, device="cuda"), torch.tensor(z, device="cuda"), rho, ws=ws,
              options=B.default_options(lanes=lanes, zero_finder=finder))
    st = B.workspace_stats(ws)
    ref = oracle.eig_all(d, z, rho, threads=16)
    tol = 16 * n * 2.0 ** -53
    for k in ("lam", "Vt"):
        assert np.max(np.abs(r[k].cpu().numpy() - ref[k]) / np.abs(ref[k])) <= tol, k
    if kind == "uniform" and finder == 0 and n > 32:
        assert st["evals_solve"] - st["screened"] - st["inferred"] <= 3 * n + st["flagged"] * 20, st
