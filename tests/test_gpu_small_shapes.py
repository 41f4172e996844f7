"""A small problem's default workspace has element buffers for the lane groups of explicit launch shapes."""
import numpy as np
import pytest
import torch

from paper_1405_7537_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs CUDA")
    return binding


@pytest.mark.parametrize("n", [33, 70, 96])
def test_eight_lane_blocks_have_buffers(B, n):
    d, z, rho = W.uniform(n, 11)
    dt, zt = torch.tensor(d, device="cuda"), torch.tensor(z, device="cuda")
    res = []
    for opt in ({}, {"lanes": 8, "warps_per_block": 8, "blocks_per_sm": 1}):
        ws = B.workspace(n, "cuda")
        r = B.eig(dt, zt, float(rho), options=B.default_options(**opt), ws=ws, check=True)
        assert B.workspace_stats(ws)["probes"] > n, opt          # screened probes need the stored elements
        res.append({k: v.cpu().numpy() for k, v in r.items() if v is not None})
    for k in res[0]:                                             # the same sums in the same order
        assert np.array_equal(res[0][k].view(np.int64), res[1][k].view(np.int64)), k
