"""The step counters hold what ran: without screens, every counted step is a binary64 evaluation."""
import numpy as np
import pytest
import torch

from paper_1405_7537_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["eig", "arrow"])
def test_unscreened_steps_are_evaluations(kind):
    """Both runs take the same bisection path.  With the screens the finishing step's bits, up to 16 for
    each eigenvalue, are among the steps that certified bounds decide (counted in evals and inferred);
    without them nothing decides a step but an evaluation, so the bits may not be counted.  On O(1) weights
    the brackets are wider than 2^16 doubles and hardly an eigenvalue is ill-conditioned, so they are at
    least 10 for nine eigenvalues in ten."""
    if not torch.cuda.is_available():
        pytest.skip("needs CUDA")
    B, n = binding, 1200
    cu = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")          # noqa: E731
    st = []
    for screen in (1, 0):
        opt = B.default_options(screen=screen)
        if kind == "eig":
            d, z, rho = W.uniform(n, 31)
            ws = B.workspace(n, "cuda")
            B.eig(cu(d), cu(z), float(rho), options=opt, ws=ws)
        else:
            d, z, alpha = W.arrowhead(n, 31)
            ws = B.arrow_workspace(n, "cuda")
            B.eig_arrowhead(cu(d), cu(z), float(alpha), options=opt, ws=ws)
        st.append(B.workspace_stats(ws))
    assert st[1]["screened"] == st[1]["inferred"] == 0
    assert st[1]["evals_solve"] <= st[0]["evals_solve"] - 9 * n, st
    # a bisection to a bracket of 2^16 doubles and about one evaluation more: at most the 53 - 16 bits of
    # a mantissa, the bracket's binades and the flagged eigenvalues' longer solves
    assert st[1]["evals_solve"] <= 42 * n + 64 * st[1]["flagged"], st
