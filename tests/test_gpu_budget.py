"""A context's memory budget: what a captured graph keeps leaves room for further graphs and datasets."""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu


def request(did, Z, depth, seed):
    return rrs.rrs_request(dataset_id=did, Z=Z.data_ptr(), n_queries=Z.shape[0], dtype=rrs.RRS_F32,
                           kind=rrs.RRS_PROJECTION, n_dirs=200, n_refinements=2, cap_shrink=0.7, seed=seed,
                           depth_out=depth.data_ptr(), count_out=None, best_out=None, round_choice_out=None,
                           precision=rrs.RRS_PREC_FP32_SIMT, reserved=0)


def test_two_graphs_and_a_dataset_within_the_budget():
    # 100 queries x 100 directions x 30,000 keys: 1.2 GB of keys a round, formed 256 MB at a time in a kept workspace
    rng = np.random.default_rng(2)
    X = torch.from_numpy(rng.standard_normal((30_000, 20), np.float32)).cuda()
    Z = torch.from_numpy(rng.standard_normal((100, 20), np.float32)).cuda()
    with rrs.Context(0) as ctx:
        want = ctx.depth(ctx.register(X), Z, rrs.RRS_PROJECTION, 200, 2, 0.7, seed=1)[0]
    stream = torch.cuda.current_stream()
    with rrs.Context(0, 1_340_000_000) as ctx:   # room for one chunk of 1 GB and no second graph
        did = ctx.register(X)
        for seed in (1, 2):
            depth = torch.empty(100, dtype=torch.float64, device="cuda")
            reqs = [request(did, Z, depth, seed)]
            rrs.rrs_depth_batched(ctx.handle, reqs, True, stream)
            rrs.rrs_check(ctx.handle, stream)
            if seed == 1:
                assert torch.equal(depth, want)
        ctx.register(torch.randn(1_000_000, 40, device="cuda"))   # 176 MB more


def test_dropped_graphs_give_their_bytes_back():
    # every kernel choice drops the cached graphs; the budget holds three such workspaces at a time
    rng = np.random.default_rng(3)
    Z = torch.from_numpy(rng.standard_normal((100, 20), np.float32)).cuda()
    depth = torch.empty(100, dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream()
    with rrs.Context(0, 900_000_000) as ctx:
        did = ctx.register(torch.from_numpy(rng.standard_normal((30_000, 20), np.float32)).cuda())
        for i in range(6):
            rrs.rrs_depth_batched(ctx.handle, [request(did, Z, depth, i)], True, stream)
            rrs.rrs_check(ctx.handle, stream)
            rrs.rrs_select_kernel(ctx.handle, did, 200, 2, 0)
