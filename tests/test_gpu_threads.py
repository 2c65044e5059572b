"""Contexts of their own on host threads of their own: what one call asks of a kernel must not reach another's launch."""
import threading

import numpy as np
import pytest
import torch

import paper_2506_08262_gb300 as rrs

pytestmark = pytest.mark.gpu


def calls(d, n, kind, nq, reps, start, out):
    """One thread: a context, a dataset and reps identical calls; the distinct results, or the error."""
    rng = np.random.default_rng(d)
    X = torch.from_numpy(rng.standard_normal((n, d), np.float32)).cuda()
    Z = torch.from_numpy(rng.standard_normal((nq, d), np.float32)).cuda()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    try:
        with torch.cuda.stream(stream), rrs.Context(0) as ctx:
            did = ctx.register(X)
            start.wait(60)
            seen = set()
            for _ in range(reps):
                depth, _, best = ctx.depth(did, Z, kind, 200, 100, 0.7, 3)
                seen.add((depth.cpu().numpy().tobytes(), best.cpu().numpy().tobytes()))
            out.append(len(seen))
    except rrs.RRSError as e:
        out.append(e)


@pytest.mark.parametrize("kind", [rrs.RRS_HALFSPACE, rrs.RRS_PROJECTION])
def test_wide_and_narrow_datasets_side_by_side(kind):
    # shared memory of a launch grows with d (directions staged) and with n (selection keys and buckets); 100 rounds a
    # call keep both threads launching
    start, out = threading.Barrier(2), []
    args = [(400, 300, kind, 4, 60, start, out), (2, 9000, kind, 4, 60, start, out)]
    threads = [threading.Thread(target=calls, args=a) for a in args]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert out == [1, 1]
