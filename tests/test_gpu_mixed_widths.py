"""A narrow FP32 halfspace request beside a dataset far wider than the halfspace kernel takes."""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu

K, R, ALPHA = 60, 2, 0.7


def data():
    rng = np.random.default_rng(7)
    return [tuple(rng.standard_normal((n, d)).astype(np.float32) for n in (300, 3)) for d in (5, 900)]


def alone(ctx, did, Z, kind):
    return ctx.depth(did, torch.from_numpy(Z).cuda(), kind, K, R, ALPHA, 4)[0].cpu().numpy()


def test_batched():
    with rrs.Context(0) as ctx:
        reqs, outs, want, keep = [], [], [], []
        for (X, Z), kind in zip(data(), (rrs.RRS_HALFSPACE, rrs.RRS_PROJECTION)):
            did = ctx.register(torch.from_numpy(X).cuda())
            Zd, out = torch.from_numpy(Z).cuda(), torch.empty(3, dtype=torch.float64, device="cuda")
            want.append(alone(ctx, did, Z, kind))
            reqs.append(rrs.rrs_request(dataset_id=did, Z=Zd.data_ptr(), n_queries=3, dtype=rrs.RRS_F32, kind=kind,
                                        n_dirs=K, n_refinements=R, cap_shrink=ALPHA, seed=4, depth_out=out.data_ptr(),
                                        count_out=None, best_out=None, round_choice_out=None,
                                        precision=rrs.RRS_PREC_FP32_SIMT, reserved=0))
            outs.append(out)
            keep.append(Zd)
        rrs.rrs_depth_batched(ctx.handle, reqs, False, torch.cuda.current_stream())
        rrs.rrs_check(ctx.handle, torch.cuda.current_stream())
        for a, b in zip(want, outs):
            assert np.array_equal(a, b.cpu().numpy())


def test_server_of_wide_slots():
    with rrs.Context(0) as ctx:
        (X, Z), _ = data()
        did = ctx.register(torch.from_numpy(X).cuda())
        want = alone(ctx, did, Z, rrs.RRS_HALFSPACE)
        srv = rrs.rrs_server_create(ctx.handle, 8, 64, 1000, torch.cuda.current_stream())
        try:
            out = np.zeros(3)
            rid = rrs.rrs_server_submit(srv, did, Z, 3, rrs.RRS_F32, rrs.RRS_HALFSPACE, K, R, ALPHA, 4, out)
            for _ in range(10):
                rrs.rrs_server_step(srv)
            torch.cuda.synchronize()
            assert rrs.rrs_server_poll(srv, rid)
        finally:
            rrs.rrs_server_destroy(srv)
        assert np.array_equal(want, out)
