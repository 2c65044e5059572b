"""Keys in device memory, small clouds and many directions: a chunk of rows is bounded by the keys launch's grid too."""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu


# a keys launch takes 65,535 tiles of 16 rows (d <= 16) or 128 rows; both cases have more rows than that in a round,
# in keys of far less than a chunk's bytes
@pytest.mark.parametrize("n,d,nq,m", [(24, 10, 8400, 125), (9, 17, 8400, 1000)])
def test_rows_beyond_one_keys_launch(n, d, nq, m):
    rng = np.random.default_rng(n)
    X = torch.from_numpy(rng.standard_normal((n, d), np.float32)).cuda()
    Z = torch.from_numpy(rng.standard_normal((nq, d), np.float32)).cuda()
    with rrs.Context(0) as ctx:
        did = ctx.register(X)
        rrs.rrs_select_kernel(ctx.handle, did, m, 1, rrs.RRS_SELECT_STREAM)
        depth, _, best = ctx.depth(did, Z, rrs.RRS_PROJECTION, m, 1, 0.7, seed=1)
        few = 50   # a query's directions depend on its place in the batch alone
        depth0, _, best0 = ctx.depth(did, Z[:few], rrs.RRS_PROJECTION, m, 1, 0.7, seed=1)
    assert torch.equal(depth[:few], depth0) and torch.equal(best[:few], best0)
    assert bool((best >= 0).all()) and bool((best < m).all())
