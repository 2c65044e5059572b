"""FP32 halfspace kernel at the edges of its tiles: rows of a task across queries, points split over CTAs.

Counts are exact on every path, so each is compared with the oracle for equality.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_08262_gb300 as rrs
import workloads

pytestmark = pytest.mark.gpu


# 256-point chunks, 64-row tasks, at least four chunks per part, 16 dims per staging step
@pytest.mark.parametrize("n", [1, 255, 257, 1025, 2047, 2048, 2305, 9001])
@pytest.mark.parametrize("d,nq,k,r,dtype", [(1, 3, 63, 1, np.float32), (2, 5, 130, 2, np.float64),
                                            (16, 1, 64, 1, np.float32), (17, 4, 150, 2, np.float32),
                                            (37, 2, 65, 1, np.float64)])
def test_counts_equal_the_oracle(n, d, nq, k, r, dtype):
    X, Z = workloads.gaussian_cloud(11, n, d, nq, dtype=dtype)
    Z[0] = X[0]   # a query that is a point of the cloud: an exact tie in every direction
    with rrs.Context(0) as ctx:
        did = ctx.register(torch.from_numpy(X).cuda())
        dep, cnt, best = ctx.depth(did, torch.from_numpy(Z).cuda(), rrs.RRS_HALFSPACE, k, r, 0.5, seed=3)
    ref = oracle.rrs(X, Z, oracle.HALFSPACE, k, r, 0.5, 3)
    assert np.array_equal(cnt.cpu().numpy(), ref["count"])
    assert np.array_equal(best.cpu().numpy(), ref["best"])
    assert np.array_equal(dep.cpu().numpy(), ref["depth"])


# the tensor-core kernel's parts: at least 8 tiles of 256 (d <= 62) or 128 points
@pytest.mark.parametrize("n", [2047, 4096, 4097, 9001, 20_001])
@pytest.mark.parametrize("d,nq,k,r,dtype", [(3, 3, 63, 1, np.float32), (62, 4, 150, 2, np.float32),
                                            (63, 2, 130, 2, np.float32), (100, 2, 65, 1, np.float64)])
def test_tensor_core_counts_equal_the_oracle(n, d, nq, k, r, dtype):
    X, Z = workloads.gaussian_cloud(12, n, d, nq, dtype=dtype)
    Z[0] = X[n - 1]
    with rrs.Context(0) as ctx:
        did = ctx.register(torch.from_numpy(X).cuda())
        dep, cnt, best = ctx.depth(did, torch.from_numpy(Z).cuda(), rrs.RRS_HALFSPACE, k, r, 0.5, seed=3,
                                   precision=rrs.RRS_PREC_SPLIT_BF16X3)
    ref = oracle.rrs(X, Z, oracle.HALFSPACE, k, r, 0.5, 3)
    assert np.array_equal(cnt.cpu().numpy(), ref["count"])
    assert np.array_equal(best.cpu().numpy(), ref["best"])
