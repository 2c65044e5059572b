"""The default selection kernels against the one that holds its keys in shared memory.

All of them select on the same FP32 keys, so depths, best directions and per-round choices are equal bit for bit:
at the edges of the point groups and bucket classes, for launches of few and of many directions (which take other
group sizes), and on data that sends directions to the iterated selection (ties, far outliers, constant clouds).
"""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu


def cloud(law, n, d, nq):
    rng = np.random.default_rng(n * 131 + d)
    if law == "normal":
        X, Z = rng.standard_normal((n, d)), 1.5 * rng.standard_normal((nq, d))
    elif law == "cauchy":
        X, Z = rng.standard_cauchy((n, d)), rng.standard_cauchy((nq, d))
    elif law == "lattice":
        X, Z = rng.integers(-1, 2, (n, d)), rng.integers(-2, 3, (nq, d))
    elif law == "shifted":   # a narrow cloud far from the origin: buckets finer than the keys
        X, Z = 4096.0 + 1e-3 * rng.standard_normal((n, d)), 4096.0 + 1e-3 * rng.standard_normal((nq, d))
    else:
        X, Z = np.ones((n, d)), rng.standard_normal((nq, d))
    return np.ascontiguousarray(X, np.float32), np.ascontiguousarray(Z, np.float32)


def run(X, Z, kind, k, r, choice):
    with rrs.Context(0) as ctx:
        did = ctx.register(torch.from_numpy(X).cuda())
        if choice:
            rrs.rrs_select_kernel(ctx.handle, did, k, r, choice)
        dep, _, best, ch = ctx.depth(did, torch.from_numpy(Z).cuda(), kind, k, r, 0.7, seed=5, rounds=True)
        return dep.cpu().numpy(), best.cpu().numpy(), ch.cpu().numpy()


@pytest.mark.parametrize("kind", [rrs.RRS_PROJECTION, rrs.RRS_ASYM_PROJECTION])
@pytest.mark.parametrize("law", ["normal", "cauchy", "lattice", "shifted", "constant"])
@pytest.mark.parametrize("n,d", [(1, 1), (2, 3), (5, 17), (31, 2), (127, 10), (1023, 16), (4000, 4), (4001, 20),
                                 (10_007, 5), (32_003, 18)])
def test_default_kernels_equal_the_resident_one(n, d, law, kind):
    for nq, k, r in ((1, 6, 2), (40, 34, 2)) if n < 10_000 else ((1, 7, 1), (5, 40, 1)):
        X, Z = cloud(law, n, d, nq)
        want = run(X, Z, kind, k, r, 1)
        for choice in (0, rrs.RRS_SELECT_STREAM) if d <= 16 else (0,):
            got = run(X, Z, kind, k, r, choice)
            for a, b in zip(want, got):
                assert np.array_equal(a, b, equal_nan=True)
