"""Selection where many keys are alike, or n outgrows the buckets: directions that need further passes.

The default kernels (keys re-formed from X, keys in device memory) against the one with its keys in shared memory, bit
for bit, in every bucket class and with enough directions for full groups; beyond what shared memory holds, against
each other and against FP64 order statistics of the same directions.
"""
import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu

PD, AP = rrs.RRS_PROJECTION, rrs.RRS_ASYM_PROJECTION


def cloud(law, n, d):
    rng = np.random.default_rng(n * 7 + d)
    X = rng.standard_normal((n, d))
    if law == "zeros":       # zero-inflated: 30% of the rows are one point
        X[rng.random(n) < 0.3] = 0.0
    elif law == "group":     # one point repeated 200 to 700 times: more than a list holds, fewer than 768
        X[rng.permutation(n)[: min(n // 3, 200 + n % 501)]] = X[0] * 0.01
    elif law == "rounded":
        X = np.round(X)
    elif law == "core":      # a dense core: 40% of the rows within 1e-4 of one another
        core = rng.random(n) < 0.4
        X[core] = 1e-4 * X[core]
    elif law == "two":       # two points, one of them in most rows
        X = np.where(rng.random((n, 1)) < 0.7, 1.0, -2.0) * np.ones((n, d))
    elif law == "tails":     # spread over many powers of ten, outlying queries and medians off centre
        X = np.exp(3.0 * X) * rng.choice([-1.0, 1.0, 1.0], (n, 1))
    elif law == "shifted":   # spread below the keys' rounding
        X = 4096.0 + 1e-3 * X
    return np.ascontiguousarray(X, np.float32)


def run(X, Z, kind, m, choice, r=2):
    with rrs.Context(0) as ctx:
        did = ctx.register(torch.from_numpy(X).cuda())
        if choice:
            rrs.rrs_select_kernel(ctx.handle, did, m * r, r, choice)
        out = ctx.depth(did, torch.from_numpy(Z).cuda(), kind, m * r, r, 0.7, seed=9, rounds=True)
        return [out[i].cpu().numpy() for i in (0, 2, 3)]


LAWS = ["zeros", "group", "rounded", "core", "two", "tails", "shifted"]


# one bucket class each (1,024 / 2,048 / 4,096 buckets), odd and even n, one and two point groups per thread
@pytest.mark.parametrize("kind", [PD, AP])
@pytest.mark.parametrize("law", LAWS)
@pytest.mark.parametrize("n,d", [(3001, 1), (900, 4), (4002, 10), (10_001, 2), (32_002, 5), (33_001, 13), (10_000, 17),
                                 (33_002, 20)])
def test_equal_to_the_resident_kernel(n, d, law, kind):
    X = cloud(law, n, d)
    Z = np.ascontiguousarray(np.vstack([X[:3], X[3:20] * 1.5 + 0.1]), np.float32)
    want = run(X, Z, kind, 35, 1)   # 700 directions a round
    for choice in (rrs.RRS_SELECT_WARP, rrs.RRS_SELECT_STREAM) if d <= 16 else (rrs.RRS_SELECT_STREAM,):
        for a, b in zip(want, run(X, Z, kind, 35, choice)):
            assert np.array_equal(a, b, equal_nan=True)


def exact_depth(X, z, u, kind):
    """FP64 depth of z along u, a device tensor of the cloud and numpy vectors."""
    y = X.double() @ torch.from_numpy(u.astype(np.float64)).cuda()
    yz = float(np.dot(z.astype(np.float64), u.astype(np.float64)))
    s = y.sort().values
    n = len(s)
    med = float(s[(n - 1) // 2] + s[n // 2]) / 2
    if kind == PD:
        s = (y - med).abs().sort().values
        num, den = abs(yz - med), float(s[(n - 1) // 2] + s[n // 2]) / 2
    else:
        s = (y - med)[y > med].sort().values
        k = len(s)
        num, den = max(yz - med, 0.0), float(s[(k - 1) // 2] + s[k // 2]) / 2 if k else 0.0
    return 1.0 if num == 0.0 else den / (den + num)


# 8,192 buckets, and n for which even they leave normal data's runs too long to list (above 1.9 million)
@pytest.mark.parametrize("kind", [PD, AP])
@pytest.mark.parametrize("law,n,d", [("normal", 130_001, 3), ("zeros", 140_000, 10), ("rounded", 131_001, 2),
                                     ("tails", 131_000, 18), ("normal", 2_300_001, 2), ("zeros", 2_000_000, 16)])
def test_beyond_shared_memory(law, n, d, kind):
    X = cloud(law, n, d)
    Z = np.ascontiguousarray(X[:4] * 1.5 + 0.05, np.float32)
    if d <= 16:
        few = run(X, Z, kind, 160, rrs.RRS_SELECT_WARP, r=1)   # 640 directions
        for a, b in zip(few, run(X, Z, kind, 160, rrs.RRS_SELECT_STREAM, r=1)):
            assert np.array_equal(a, b)
    m = 6
    U = np.random.default_rng(3).standard_normal((4 * m, d)).astype(np.float32)
    U = np.ascontiguousarray(U / np.linalg.norm(U, axis=1, keepdims=True).astype(np.float32))
    depth = torch.empty(4 * m, dtype=torch.float64, device="cuda")
    with rrs.Context(0) as ctx:
        Xd = torch.from_numpy(X).cuda()
        did = ctx.register(Xd)
        rrs.rrs_debug_round_depths(ctx.handle, did, torch.from_numpy(Z).cuda(), 4, rrs.RRS_F32, kind, m,
                                   torch.from_numpy(U).cuda(), rrs.RRS_PREC_FP32_SIMT, depth)
    want = [exact_depth(Xd, Z[i // m], U[i], kind) for i in range(4 * m)]
    # the parity bound of projection depths: FP32 keys choose the points, FP64 forms the depth
    assert np.allclose(depth.cpu().numpy(), want, rtol=1e-5, atol=1e-12)


# the allocation-free call has neither columns nor keys in memory
@pytest.mark.parametrize("kind", [PD, AP])
@pytest.mark.parametrize("law,n,d", [("zeros", 2003, 5), ("rounded", 20_001, 2), ("core", 33_000, 9)])
def test_allocation_free(law, n, d, kind):
    X = cloud(law, n, d)
    Z = np.ascontiguousarray(X[:8] * 1.5 + 0.1, np.float32)
    want = run(X, Z, kind, 40, 1)[0]
    Xd, Zd = torch.from_numpy(X).cuda(), torch.from_numpy(Z).cuda()
    depth = torch.empty(8, dtype=torch.float64, device="cuda")
    count = torch.empty(8, dtype=torch.int64, device="cuda")
    rrs.rrs_depth_noalloc(Xd, n, d, rrs.RRS_F32, Zd, 8, kind, 80, 2, 0.7, 9, depth, count, torch.cuda.current_stream())
    assert np.array_equal(depth.cpu().numpy(), want, equal_nan=True)
