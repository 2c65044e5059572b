"""FP32 halfspace: a query far from the data must not widen the near-tie bands of the queries beside it."""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu


def bands(ctx, did, Z, m, U):
    """Counts and near ties per query of one call on caller-supplied directions (m per query)."""
    nq = Z.shape[0]
    depth = torch.empty(nq * m, dtype=torch.float64, device="cuda")
    count = torch.empty(nq * m, dtype=torch.int64, device="cuda")
    band = torch.empty(nq, dtype=torch.int64, device="cuda")
    rrs.rrs_debug_round_depths(ctx.handle, did, torch.from_numpy(Z).cuda(), nq, rrs.RRS_F32, rrs.RRS_HALFSPACE, m,
                               U[: nq * m].contiguous(), rrs.RRS_PREC_FP32_SIMT, depth, count, band)
    return count.cpu().numpy().reshape(nq, m), band.cpu().numpy()


# 20 directions a query: three queries share a task of 64 rows
@pytest.mark.parametrize("n,d", [(5000, 20), (257, 3)])
def test_neighbours_keep_their_bands(n, d):
    rng = np.random.default_rng(d)
    X, Z = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((3, d)).astype(np.float32)
    far = Z.copy()
    far[0] *= 1e6
    m = 20
    U = torch.randn(3 * m, d, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    U /= U.norm(dim=1, keepdim=True)
    with rrs.Context(0) as ctx:
        did = ctx.register(torch.from_numpy(X).cuda())
        count, near = bands(ctx, did, Z, m, U)
        count_far, near_far = bands(ctx, did, far, m, U)
    assert np.array_equal(count[1:], count_far[1:])
    # a row's own bound is at most the largest of its task's rows, up to a rounding of the bound
    assert (near_far[1:] <= near[1:] + 2).all()
