"""Timing cases of the depth library: what its users have it do, through its public entry points.

``listed()`` names the cases, ``draw(rng)`` gives another of the same ranges, ``prepare(case, seed)`` makes
the inputs and the handle a program keeps (a context with its registered datasets, a server), ``run(state)``
is one pass, ``work(case)`` what a pass cannot do without, and ``exact(case, seed)`` the same depths in 64
bits from plain torch: the direction stream of the written formula (Philox4x32-10, one FP32 operation per
step), FP64 projections, sorted order statistics.

A case's ``entry`` is the way in:

* ``tensors``   ``Context.depth``: queries and results are CUDA tensors, the call every torch program makes;
* ``host``      ``rrs_depth`` with host queries and host results, the whole call as a C program sees it;
* ``noalloc``   ``rrs_depth_noalloc``: no registered dataset, no allocation;
* ``batched``   ``rrs_depth_batched`` over many datasets, replayed as a graph;
* ``serving``   the continuous-batching server: submit a burst, step until every request is done.
"""
import math

import numpy as np
import torch

import paper_2506_08262_gb300 as rrs

KINDS = {"halfspace": rrs.RRS_HALFSPACE, "projection": rrs.RRS_PROJECTION, "asymmetric": rrs.RRS_ASYM_PROJECTION}
PREC = {"fp32": rrs.RRS_PREC_FP32_SIMT, "tc": rrs.RRS_PREC_SPLIT_BF16X3}


def _one(name, entry, kind, n, d, nq, k, r, alpha, law, dtype="f32", prec="fp32"):
    c = {"entry": entry, "kind": kind, "n": n, "d": d, "nq": nq, "k": k, "r": r, "alpha": alpha, "law": law,
         "dtype": dtype, "prec": prec}
    return {"name": name, **c} if name else c


def _many(name, entry, datasets, n_lo, n_hi, d_lo, d_hi, requests, q_hi, k, r, mix):
    c = {"entry": entry, "datasets": datasets, "n_lo": n_lo, "n_hi": n_hi, "d_lo": d_lo, "d_hi": d_hi,
         "requests": requests, "q_hi": q_hi, "k": k, "r": r, "alpha": 0.9, "mix": mix}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the two-dimensional halfspace workload on FP64 data: a short call, bound by its launches
        _one("halfspace_2d", "tensors", "halfspace", 1000, 2, 100, 1000, 10, 0.5, "normal", dtype="f64"),
        # one query point at a time, as the paper times its grid: the latency of an interactive call
        _one("projection_one_point", "tensors", "projection", 10_000, 5, 1, 1000, 10, 0.9, "toeplitz"),
        # the headline workload: outlier scores of a batch against a contaminated cloud
        _one("projection_10d", "tensors", "projection", 10_000, 10, 1000, 1000, 20, 0.7, "mixture"),
        # its asymmetric half, from host buffers and back, as a C program calls it
        _one("asymmetric_10d_host", "host", "asymmetric", 10_000, 10, 1000, 1000, 20, 0.7, "mixture"),
        # the large halfspace workload on the tensor cores, a tenth of its queries
        _one("halfspace_50d_tc", "tensors", "halfspace", 100_000, 50, 1000, 2000, 20, 0.9, "student3", prec="tc"),
        # the same cloud on the FP32 path, which every d and the servers without tensor cores take
        _one("halfspace_50d_fp32", "tensors", "halfspace", 100_000, 50, 100, 2000, 20, 0.9, "student3"),
        # FP64 data of the widest class of dimensions, an odd number of points
        _one("halfspace_100d_tc_f64", "tensors", "halfspace", 33_333, 100, 256, 1000, 10, 0.9, "student3",
             dtype="f64", prec="tc"),
        # the timing grid's batch of 32 points at d = 50, many directions each
        _one("projection_50d_grid", "tensors", "projection", 10_000, 50, 32, 10_000, 10, 0.9, "toeplitz"),
        # the ranking study: heavy tails, a cloud far beyond shared memory, queries from the cloud
        _one("ranking_100d", "tensors", "projection", 100_000, 100, 10, 10_000, 40, 0.9, "student5"),
        # a plug-in that may not allocate scores a few points of a small cloud
        _one("noalloc_3d", "noalloc", "asymmetric", 2_003, 3, 17, 500, 5, 0.8, "normal"),
        # many uneven datasets and kinds in shared launches, replayed as a graph
        _many("batched_mixed", "batched", 32, 500, 50_000, 5, 100, 32, 64, 1000, 10, 4),
        # a burst of requests to resident datasets, kinds 50/30/20, served to completion
        _many("serving_burst", "serving", 16, 500, 50_000, 5, 100, 40, 256, 1000, 10, 5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["tensors", "tensors", "tensors", "host", "noalloc", "batched", "serving"])
    if form == "batched":
        return _many("", form, rng.randint(3, 24), 500, 20_000, 5, 100, rng.randint(3, 24), _log_int(rng, 2, 48),
                     rng.choice([500, 1000]), rng.choice([5, 10]), rng.randrange(1 << 20))
    if form == "serving":
        return _many("", form, rng.randint(2, 12), 500, 20_000, 5, 100, rng.randint(4, 32), _log_int(rng, 2, 128),
                     1000, 10, rng.randrange(1 << 20))
    kind = rng.choice(sorted(KINDS))
    dtype = rng.choice(["f32", "f32", "f64"])
    alpha = rng.choice([0.5, 0.7, 0.8, 0.9])
    r = rng.choice([1, 5, 10, 20])
    law = rng.choice(["normal", "toeplitz", "student3", "student5", "mixture"])
    if form == "noalloc":
        return _one("", form, kind, _log_int(rng, 200, 20_000), _log_int(rng, 2, 20), _log_int(rng, 1, 32),
                    _log_int(rng, 100, 1000), r, alpha, law, dtype)
    n, d, nq, k = _log_int(rng, 500, 100_000), _log_int(rng, 2, 120), _log_int(rng, 1, 1000), _log_int(rng, 100, 5000)
    prec = rng.choice(["tc", "fp32"]) if kind == "halfspace" else "fp32"
    # no dearer than the largest listed pass
    most = 1e13 if prec == "tc" else 4e11
    while nq > 1 and n * nq * k * (d + 30) > most:
        nq = max(1, nq * 3 // 4)
    while n > 500 and n * nq * k * (d + 30) > most:
        n = n * 3 // 4
    return _one("", form, kind, n, d, nq, k, r, alpha, law, dtype, prec)


# ---- inputs -------------------------------------------------------------------------------------


def _rows(gen, law, n, d, A):
    """n rows of a law, FP64 on the GPU."""
    z = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)
    if law == "mixture":   # 95% N(0, I), 5% N(6*1, I), shuffled
        out = torch.rand(n, 1, generator=gen, device="cuda", dtype=torch.float64) < 0.05
        return z(n, d) + 6.0 * out
    if law == "student3":  # independent Student-t(3) coordinates, mapped by a random SPD square root
        return z(n, d) / torch.sqrt((z(n, d) ** 2 + z(n, d) ** 2 + z(n, d) ** 2) / 3) @ A
    if law == "student5":  # multivariate Student-t(5) of Toeplitz scatter
        return z(n, d) @ A / torch.sqrt((z(n, 5) ** 2).sum(1, keepdim=True) / 5)
    return z(n, d) @ A if A is not None else z(n, d)


def _matrix(rng, law, d):
    if law == "toeplitz" or law == "student5":
        i = np.arange(d)
        A = np.linalg.cholesky(2.0 ** -np.abs(i[:, None] - i[None, :])).T
    elif law == "student3" or law == "spd":   # eigenvalues log-uniform in [0.1, 10], Haar eigenvectors
        Q, R = np.linalg.qr(rng.standard_normal((d, d)))
        Q = Q * np.sign(np.diag(R))
        A = (Q * np.exp(0.5 * rng.uniform(math.log(0.1), math.log(10.0), d))) @ Q.T
    else:
        return None
    return torch.from_numpy(np.ascontiguousarray(A)).cuda()


def _cloud(c, seed):
    """The cloud and the query batch of a single-dataset case, in its type, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    A = _matrix(np.random.default_rng(seed), c["law"], c["d"])
    dt = torch.float32 if c["dtype"] == "f32" else torch.float64
    X = _rows(gen, c["law"], c["n"], c["d"], A).to(dt).contiguous()
    if c["law"] == "mixture":
        Z = torch.rand(c["nq"], c["d"], generator=gen, device="cuda", dtype=torch.float64) * 8 - 4
    elif c["law"] == "student5":   # ranking: points of the cloud itself
        Z = X[torch.randint(c["n"], (c["nq"],), generator=gen, device="cuda")]
    else:
        Z = _rows(gen, c["law"], c["nq"], c["d"], A)
        if c["law"] == "normal":
            Z = 1.5 * Z
    return X, Z.to(dt).contiguous()


def _mix(c):
    """Sizes of a many-dataset case: [(n, d)], [(dataset, kind, queries)]."""
    rng = np.random.default_rng(c["mix"])
    shapes = [(int(round(math.exp(rng.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]))))),
               int(rng.integers(c["d_lo"], c["d_hi"] + 1))) for _ in range(c["datasets"])]
    reqs = []
    for i in range(c["requests"]):
        if c["entry"] == "batched":
            reqs.append((i % c["datasets"], int(rng.integers(0, 3)), int(rng.integers(1, c["q_hi"] + 1))))
        else:
            reqs.append((int(rng.integers(0, c["datasets"])), int(rng.choice(3, p=[0.5, 0.3, 0.2])),
                         int(round(math.exp(rng.uniform(0.0, math.log(c["q_hi"])))))))
    return shapes, reqs


class _State:
    """What a program keeps: the context (closed with the state), its datasets, queries and result buffers."""

    def __init__(self):
        self.ctx = None
        self.server = None

    def __del__(self):
        if self.server:
            rrs.rrs_server_destroy(self.server)
        if self.ctx:
            self.ctx.close()


def prepare(case, seed):
    s = _State()
    s.case, s.seed = case, seed
    if "mix" not in case:
        s.X, s.Z = _cloud(case, seed)
        s.kind, s.prec = KINDS[case["kind"]], PREC[case["prec"]]
        nq = case["nq"]
        if case["entry"] == "noalloc":
            s.depth = torch.empty(nq, dtype=torch.float64, device="cuda")
            s.count = torch.empty(nq, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            return s
        s.ctx = rrs.Context(0)
        s.did = s.ctx.register(s.X)
        if case["entry"] == "host":
            s.Z = s.Z.cpu().pin_memory()
            s.depth = torch.empty(nq, dtype=torch.float64, pin_memory=True)
            s.count = torch.empty(nq, dtype=torch.int64, pin_memory=True)
            s.best = torch.empty(nq, dtype=torch.int32, pin_memory=True)
        return s
    shapes, reqs = _mix(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    s.ctx = rrs.Context(0)
    clouds = []
    for n, d in shapes:
        A = _matrix(rng, "spd", d)
        mu = torch.from_numpy(rng.uniform(-5.0, 5.0, d)).cuda()
        X = (_rows(gen, "", n, d, A) + mu).float().contiguous()
        clouds.append((s.ctx.register(X), A, mu, d))
    s.reqs = []
    for ds, kind, nq in reqs:
        did, A, mu, d = clouds[ds]
        s.reqs.append((did, kind, nq, (_rows(gen, "", nq, d, A) + mu).float().contiguous()))
    if case["entry"] == "batched":
        s.depth = [torch.empty(nq, dtype=torch.float64, device="cuda") for _, _, nq, _ in s.reqs]
        s.best = [torch.empty(nq, dtype=torch.int32, device="cuda") for _, _, nq, _ in s.reqs]
        s.desc = [rrs.rrs_request(dataset_id=did, Z=Z.data_ptr(), n_queries=nq, dtype=rrs.RRS_F32, kind=kind,
                                  n_dirs=case["k"], n_refinements=case["r"], cap_shrink=case["alpha"], seed=seed,
                                  depth_out=dep.data_ptr(), count_out=None, best_out=best.data_ptr(),
                                  round_choice_out=None, precision=PREC["tc"] if kind == 0 else PREC["fp32"], reserved=0)
                  for (did, kind, nq, Z), dep, best in zip(s.reqs, s.depth, s.best)]
        torch.cuda.synchronize()
        return s
    s.reqs = [(did, kind, nq, Z.cpu().numpy()) for did, kind, nq, Z in s.reqs]
    s.depth = [np.zeros(nq) for _, _, nq, _ in s.reqs]
    m = -(-case["k"] // case["r"])
    s.server = rrs.rrs_server_create(s.ctx.handle, 4096, m, 100, torch.cuda.current_stream(), PREC["tc"])
    return s


# ---- one pass -----------------------------------------------------------------------------------


def run(s):
    c = s.case
    if c["entry"] == "tensors":
        depth, count, best = s.ctx.depth(s.did, s.Z, s.kind, c["k"], c["r"], c["alpha"], s.seed, s.prec)
        return {"depth": depth, "count": count, "best": best}
    if c["entry"] == "host":
        rrs.rrs_depth(s.ctx.handle, s.did, s.Z, c["nq"], s.ctx._dtype_code(s.Z), False, s.kind, c["k"], c["r"],
                      c["alpha"], s.seed, s.prec, s.depth, s.count, s.best, None, False, torch.cuda.current_stream())
        return {"depth": s.depth, "count": s.count, "best": s.best}
    if c["entry"] == "noalloc":
        code = rrs.RRS_F32 if c["dtype"] == "f32" else rrs.RRS_F64
        rrs.rrs_depth_noalloc(s.X, c["n"], c["d"], code, s.Z, c["nq"], s.kind, c["k"], c["r"], c["alpha"], s.seed,
                              s.depth, s.count, torch.cuda.current_stream())
        return {"depth": s.depth, "count": s.count}
    if c["entry"] == "batched":
        rrs.rrs_depth_batched(s.ctx.handle, s.desc, True, torch.cuda.current_stream())
        return {"depth": s.depth, "best": s.best}
    ids = [rrs.rrs_server_submit(s.server, did, Z, nq, rrs.RRS_F32, kind, c["k"], c["r"], c["alpha"], s.seed, dep)
           for (did, kind, nq, Z), dep in zip(s.reqs, s.depth)]
    while ids:
        rrs.rrs_server_step(s.server)
        ids = [i for i in ids if not rrs.rrs_server_poll(s.server, i)]
    return {"depth": s.depth}


# ---- what a pass cannot do without ----------------------------------------------------------------


def _pair_flops(kind, d, tc):
    # halfspace: the product (three BF16 products on the tensor cores) and a comparison; projection depths:
    # the product, and a subtraction and a comparison for each of the two medians
    return (6 * d if tc else 2 * d) + 2 if kind == 0 else 2 * d + 4


def work(case):
    if "mix" not in case:
        m = -(-case["k"] // case["r"])
        pairs = case["n"] * case["nq"] * m * case["r"]
        size = 4 if case["dtype"] == "f32" else 8
        kind = KINDS[case["kind"]]
        return {"bytes": (case["n"] + case["nq"]) * case["d"] * size + 20 * case["nq"],
                "flops": pairs * _pair_flops(kind, case["d"], case["prec"] == "tc")}
    shapes, reqs = _mix(case)
    m = -(-case["k"] // case["r"])
    return {"bytes": sum(4 * n * d for n, d in shapes) + sum(nq * (4 * shapes[ds][1] + 12) for ds, _, nq in reqs),
            "flops": sum(shapes[ds][0] * nq * m * case["r"] * _pair_flops(kind, shapes[ds][1], True)
                         for ds, kind, nq in reqs)}


# ---- the same depths in 64 bits ---------------------------------------------------------------------

_MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c0, c1, c2, c3


def _unif(w):
    return (2 * (w >> 9) + 1).float() * 2.0 ** -24


def _f(v):
    return float(np.float32(v))


def _log(a):
    bits = a.view(torch.int32)
    e = ((bits >> 23) & 0xFF) - 127
    f = ((bits & 0x007FFFFF) | 0x3F800000).view(torch.float32)
    big = f > _f(1.41421356)
    f, e = torch.where(big, f * 0.5, f), torch.where(big, e + 1, e)
    s = (f - 1.0) / (f + 1.0)
    z = s * s
    p = torch.full_like(z, _f(1 / np.float32(13)))
    for q in (11, 9, 7, 5, 3):
        p = p * z + _f(1 / np.float32(q))
    t = 2.0 * s
    ef = e.float()
    return ef * 0.693145751953125 + (ef * _f(1.42860682e-06) + (t + t * (z * p)))


def _sincos(a):
    """sin and cos of (pi/2) a, a in [0, 4)."""
    q = a.to(torch.int32)
    r = a - q.float()
    up = r > 0.5
    r, q = torch.where(up, r - 1.0, r), torch.where(up, q + 1, q)
    x = r * _f(1.57079637)
    z = x * x
    ps = torch.full_like(z, _f(1 / np.float32(362880)))
    for v in (-1 / np.float32(5040), 1 / np.float32(120), -1 / np.float32(6)):
        ps = ps * z + _f(v)
    sx = x + x * (z * ps)
    pc = torch.full_like(z, _f(-1 / np.float32(3628800)))
    for v in (1 / np.float32(40320), -1 / np.float32(720), 1 / np.float32(24), -0.5):
        pc = pc * z + _f(v)
    cx = 1.0 + z * pc
    q = q & 3
    return (torch.where(q == 0, sx, torch.where(q == 1, cx, torch.where(q == 2, -sx, -cx))),
            torch.where(q == 0, cx, torch.where(q == 1, -sx, torch.where(q == 2, -cx, sx))))


def _gaussians(seed, rnd, q, j, cnt):
    """(queries, directions, cnt) Gaussians of the stream."""
    nb = -(-cnt // 4)
    b = torch.arange(nb, device=q.device)[None, None, :]
    o = torch.zeros_like(b)
    w = _philox(b + 0 * j[None, :, None] + 0 * q[:, None, None], j[None, :, None] + o, torch.full_like(b, rnd),
                q[:, None, None] + o, seed)
    out = []
    for wa, wb in ((w[0], w[1]), (w[2], w[3])):
        R = torch.sqrt(-2.0 * _log(_unif(wa)))
        s, c = _sincos(4.0 * _unif(wb))
        out += [R * c, R * s]
    return torch.stack(out, -1).flatten(2)[..., :cnt]


def _seq_dot(a, b):
    s = a[..., 0] * b[..., 0]
    for i in range(1, a.shape[-1]):
        s = s + a[..., i] * b[..., i]
    return s


def _directions(seed, rnd, q, m, d, alpha, pole):
    """The m FP32 directions of round rnd (0-based) of each query, (queries, m, d)."""
    j = torch.arange(m, device=q.device)
    if rnd == 0:
        g = _gaussians(seed, 0, q, j, d)
        return g / torch.sqrt(0.0 + _seq_dot(g, g))[..., None]
    ap = np.float32(1.0)
    for _ in range(rnd):
        ap = np.float32(ap * np.float32(alpha))
    one = torch.ones(1, 1, dtype=torch.int64, device=q.device)
    w = _philox(one * _MASK, j[None, :] * one, one * rnd, q[:, None] * one, seed)
    st, ct = _sincos(_unif(w[0] + 0 * j[None, :]) * float(ap))
    u = ct[..., None]
    if d > 1:
        g = _gaussians(seed, rnd, q, j, d - 1)
        u = torch.cat([u, st[..., None] * (g / torch.sqrt(0.0 + _seq_dot(g, g))[..., None])], -1)
    v = -pole
    v[:, 0] = 1.0 - pole[:, 0]
    vv = _seq_dot(v, v)
    lam = (2.0 * _seq_dot(v[:, None, :].expand_as(u), u)) / vv[:, None]
    return torch.where(vv[:, None, None] == 0, u, u - lam[..., None] * v[:, None, :])


def _univariate(kind, y, yz):
    """Depth of yz (m,) in the rows of y (m, n), FP64."""
    n = y.shape[1]
    if kind == 0:
        return torch.minimum((y <= yz[:, None]).sum(1), (y >= yz[:, None]).sum(1)).double() / n
    k1, k2 = (n - 1) // 2, n // 2
    s = y.sort(1).values
    med = (s[:, k1] + s[:, k2]) * 0.5
    if kind == 1:
        t = (s - med[:, None]).abs().sort(1).values
        spread, num = (t[:, k1] + t[:, k2]) * 0.5, (yz - med).abs()
    else:
        le = (s <= med[:, None]).sum(1)
        npos = n - le
        at = lambda i: s.gather(1, i.clamp(0, n - 1)[:, None])[:, 0] - med
        spread = torch.where(npos > 0, (at(le + (npos - 1).clamp(min=0) // 2) + at(le + npos // 2)) * 0.5, 0.0 * med)
        num = (yz - med).clamp(min=0.0)
    return torch.where(spread > 0, spread / (spread + num), (num == 0).double())


def exact(case, seed):
    if "mix" in case:
        return None
    kind = KINDS[case["kind"]]
    m, r, d = -(-case["k"] // case["r"]), case["r"], case["d"]
    pairs = case["n"] * case["nq"] * m * r
    if pairs * d > 1.5e12 if kind == 0 else pairs > 4e9:   # tens of seconds
        return None
    X, Z = _cloud(case, seed)
    X, Z, alpha = X.double(), Z.double(), np.float32(case["alpha"])
    nq = case["nq"]
    pole = torch.zeros(nq, d, device="cuda")
    pole[:, 0] = 1.0
    best = torch.ones(nq, dtype=torch.float64, device="cuda")
    step = max(1, int(4e8 // (m * max(case["n"], d))))   # queries at a time
    for rnd in range(r):
        for q0 in range(0, nq, step):
            q = torch.arange(q0, min(nq, q0 + step), device="cuda")
            U = _directions(seed, rnd, q, m, d, alpha, pole[q].clone())
            Ud = U.double()
            if kind == 0:   # of the differences, so that a query that is a point of the cloud ties with it
                dep = torch.stack([_univariate(0, Ud[i] @ (X - Z[q0 + i]).T, torch.zeros_like(Ud[i, :, 0]))
                                   for i in range(len(q))])
            else:
                yz = (Ud * Z[q][:, None, :]).sum(-1)
                dep = _univariate(kind, Ud.flatten(0, 1) @ X.T, yz.flatten()).view(len(q), m)
            val, at = dep.min(1)
            take = val < best[q]
            best[q] = torch.where(take, val, best[q])
            pole[q] = torch.where(take[:, None], U[torch.arange(len(q), device="cuda"), at], pole[q])
    out = {"depth": best, "count": None}
    if case["entry"] != "noalloc":
        out["best"] = None
    return out
