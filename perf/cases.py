"""What is measured: calls that users of the PM-LSH library make, over the
sizes that the repository's data sets, tests and benchmark span.

The data are Gaussian mixtures like those of `datagen` (cluster centres
N(0, 10^2 I), a scale per cluster, queries from the same mixture), drawn on
the GPU.  The projection matrix is the caller's own (the `proj` build option),
so that `exact` can follow every algorithm in FP64 with plain PyTorch.

Ranges: n 10,000 to 1,000,000 points, d 64 to 960 (odd ones too), 1 to 10,000
queries per call, k 1 to 100 neighbours (closest pairs: 10 to 1,000), c 1.2
to 2, the paper's budget beta = 0.2809 and small ones, m 8 to 16 projections,
leaves of 16 to 512 points, each precision mode, with and without statistics,
rows in device and in host memory.
"""
import math

import numpy as np
import torch

import paper_2107_05537_gb300 as pm

PREC = {"fp32": pm.PMLSH_FP32_PLAIN, "tensor": pm.PMLSH_BF16_TENSOR, "verify": pm.PMLSH_BF16_VERIFY,
        "rerank": pm.PMLSH_BF16_RERANK}

BASE = dict(n=100_000, d=128, clusters=100, sigma_lo=0.5, sigma_hi=2.0, aniso=False, nq=1000, k=10, m=15, leaf=256,
            c=1.5, beta=0.2809, precision="fp32", stats=True, host=False, r=0.0, planted=0)


def listed():
    def case(name, op, **kw):
        return dict(BASE, name=name, op=op, **kw)

    return [
        # one lookup by an interactive program: host row in, host results out,
        # default options, the small data set of the parity tests (latency)
        case("one_query", "knn", n=10_000, clusters=50, sigma_lo=1.0, sigma_hi=1.0, nq=1, host=True),
        # the paper's query experiment on its smallest set: 200 queries, k = 50, at the
        # Audio shape (54K x 192), default options
        case("audio", "knn", n=54_387, d=192, nq=200, k=50),
        # an odd-sized batch from a service with its own settings: ragged row
        # length, fewer projections, smaller leaves, ids and distances only
        case("ragged", "knn", n=199_999, d=100, clusters=333, nq=1001, k=7, m=12, leaf=128, precision="tensor",
             stats=False),
        # the throughput workload of the benchmark: a large batch, ids,
        # distances and error bounds
        case("throughput", "knn", n=1_000_000, clusters=1000, nq=10_000, k=50, precision="tensor", stats=False),
        # an offline job with the default options (FP32 count, per-query statistics)
        case("default_batch", "knn", n=300_000, clusters=300, nq=5000, k=10),
        # high-dimensional descriptors (the GIST shape), BF16 first pass and FP32 rerank
        case("gist", "knn", n=200_000, d=960, clusters=200, sigma_lo=1.0, sigma_hi=1.0, aniso=True, nq=1000, k=10,
             precision="rerank", stats=False),
        # a small candidate budget: stop rule 2 cuts the range sets of many queries
        case("budget", "knn", n=300_000, d=96, clusters=100, nq=2000, k=10, beta=0.01, precision="tensor", stats=False),
        # near-duplicate lookups at a fixed radius (Algorithm 1)
        case("radius", "rcbc", n=100_000, nq=1000, k=1, r=9.0, precision="tensor"),
        # a serving process: 24 requests of 1 to 1,024 rows with k of 1, 10 and
        # 100 in flight at once, host rows in and host results out
        case("serve", "serve", n=200_000, d=256, clusters=200, sigma_lo=1.0, sigma_hi=1.0, nq=1024, k=100,
             precision="tensor", stats=False),
        # duplicate detection: the ten closest pairs of a set with five planted
        # near-duplicates, radius filtering with the calibrated gamma
        case("closest_pairs", "cp", n=100_000, d=512, clusters=500, sigma_lo=1.0, sigma_hi=1.0, leaf=16, planted=5),
        # the paper's closest-pair experiment (k = 10^3) at the MNIST shape
        # (60K x 784), branch and bound
        case("branch_and_bound", "bnb", n=60_000, d=784, k=1000, leaf=16, sigma_lo=1.0, sigma_hi=1.0),
        # (re)building the index when the data set changes, and reading it back
        case("build", "build", n=100_000),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["knn", "knn", "knn", "knn", "rcbc", "serve", "cp", "bnb", "build"])
    c = dict(BASE, op=op)
    c["d"] = spread(64, 960)
    c["m"] = rng.choice([8, 10, 12, 15, 15, 16])
    lo = rng.choice([0.5, 1.0])
    c["sigma_lo"], c["sigma_hi"] = lo, rng.choice([lo, 2.0])
    if op in ("cp", "bnb"):
        c["m"], c["leaf"] = 15, rng.choice([16, 24, 32])
        c["n"] = spread(10_000, min(100_000, 30_000_000 // c["d"]) if op == "cp" else 45_000)
        c["sigma_lo"] = c["sigma_hi"] = 1.0
        c["k"] = spread(10, 1000) if op == "bnb" else 10
        c["planted"] = 5 if op == "cp" else 0
        c["clusters"] = max(20, c["n"] // rng.choice([100, 200, 400]))
        return c
    # up to 128 M coordinates; a build alone up to the listed one's 12.8 M
    c["n"] = spread(10_000, min(1_000_000, 128_000_000 // c["d"]))
    if op == "build":
        c["n"] = spread(10_000, min(100_000, 12_800_000 // c["d"]))
    if op == "serve":
        c["n"] = min(c["n"], 400_000)
    c["clusters"] = max(20, c["n"] // rng.choice([200, 600, 1000]))
    c["leaf"] = rng.choice([64, 128, 200, 256, 512])
    c["precision"] = rng.choice(["fp32", "tensor", "verify", "rerank"])
    c["stats"] = rng.random() < 0.5
    c["host"] = rng.random() < 0.3
    c["nq"] = spread(1, min(10_000, 1_280_000_000 // (c["n"] * max(1, c["d"] // 128))))
    c["k"] = spread(1, 100)
    c["c"] = rng.choice([1.2, 1.5, 1.5, 2.0])
    c["beta"] = rng.choice([0.2809, 0.2809, 0.05, 0.01])
    if op == "serve":
        c.update(nq=1024, k=100, stats=False, precision=rng.choice(["fp32", "tensor"]), host=False)
    if op == "rcbc":
        c.update(k=1, stats=True, r=round(rng.uniform(0.5, 1.2) * math.sqrt(c["d"]), 3))
    return c


# --------------------------------------------------------------------- inputs

def _data(case, seed):
    """(X [n][d], Q [nq][d], projection A [m][d]) on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, d, cl = case["n"], case["d"], case["clusters"]
    centres = torch.randn(cl, d, generator=g, device="cuda") * 10.0
    lo, hi = case["sigma_lo"], case["sigma_hi"]
    scale = lo + (hi - lo) * torch.rand(cl, generator=g, device="cuda")
    # anisotropic clusters: covariance eigenvalues i^-1
    shape = torch.arange(1, d + 1, device="cuda").float().rsqrt() if case["aniso"] else torch.ones(d, device="cuda")

    def members(count):
        lab = torch.randint(0, cl, (count,), generator=g, device="cuda")
        z = torch.randn(count, d, generator=g, device="cuda")
        return z.mul_(shape).mul_(scale[lab, None]).add_(centres[lab])

    X = members(n)
    if case["planted"]:
        at = torch.randperm(n, generator=g, device="cuda")[:2 * case["planted"]].view(2, -1)
        u = torch.randn(case["planted"], d, generator=g, device="cuda")
        X[at[1]] = X[at[0]] + 0.01 * u / u.norm(dim=1, keepdim=True)
    Q = members(case["nq"])
    A = torch.randn(case["m"], d, generator=g, device="cuda")
    return X, Q, A


def _requests(case, Q, seed):
    """The serving case's requests: (rows, k), sizes spread evenly over their logarithm."""
    rng = np.random.default_rng(seed)
    Qh = Q.cpu().numpy()
    reqs = []
    for i in range(24):
        size = int(round(case["nq"] ** ((i * 7 % 24) / 23.0)))
        first = int(rng.integers(0, case["nq"] - size + 1))
        reqs.append((Qh[first:first + size], (1, 10, case["k"])[i % 3]))
    return reqs


def prepare(case, seed):
    X, Q, A = _data(case, seed)
    torch.cuda.synchronize()
    s = dict(case=case)
    if case["op"] == "build":
        s.update(X=X, A=A)
        return s
    s["ix"] = pm.Index(X, m=case["m"], leaf_size=case["leaf"], proj=A)
    if case["op"] == "serve":
        s["reqs"] = _requests(case, Q, seed)
        s["server"] = pm.Server(s["ix"])
    else:
        s["Q"] = Q.cpu().numpy() if case["host"] else Q
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "build":
        ix = pm.Index(s["X"], m=case["m"], leaf_size=case["leaf"], proj=s["A"])
        # coordinates and leaf hierarchy; as many leaves and nodes as the data
        # give, in arrays of one size
        lay = ix.layout()
        out = dict(projected=ix.projected(), perm=lay["perm"])
        for f in ("leaf_off", "node_lo", "node_hi", "node_left", "node_right"):
            out[f] = np.full(2 * ix.n, -2, lay[f].dtype)
            out[f][:len(lay[f])] = lay[f]
        ix.close()
        return out
    ix = s["ix"]
    if op == "knn":
        r = ix.knn(s["Q"], k=case["k"], c=case["c"], beta=case["beta"], precision=PREC[case["precision"]],
                   with_stats=case["stats"])
        out = dict(ids=r["ids"], dists=r["dists"], err=r["err"])
        if case["stats"]:
            # the algorithm's trace; the other statistics count the work done
            out["stats"] = {f: r["stats"][f] for f in ("rounds", "rule", "ncand", "r")}
        return out
    if op == "rcbc":
        r = ix.rcbc(s["Q"], case["r"], c=case["c"], beta=case["beta"], precision=PREC[case["precision"]])
        return dict(ids=r["ids"], dists=r["dists"], stats=r["stats"])
    if op == "serve":
        sv = s["server"]
        tickets = [sv.submit(q, k=k, c=case["c"], beta=case["beta"], precision=PREC[case["precision"]])
                   for q, k in s["reqs"]]
        return [sv.wait(t) for t in tickets]
    if op == "cp":
        r = ix.closest_pairs(k=case["k"], c=case["c"])
    else:
        r = ix.closest_pairs_bnb(k=case["k"])
    return dict(pairs=r["pairs"], dists=r["dists"], count=r["stats"]["count"])


def work(case):
    """What a pass cannot do without: the queries in and the results out; per
    returned neighbour its row and distance; the projections.  A build and a
    closest-pair call read every row once; branch and bound computes the
    distance of each of its T pairs."""
    n, d, nq, k, m, op = (case[f] for f in ("n", "d", "nq", "k", "m", "op"))
    if op == "build":
        return dict(bytes=4 * n * d + 8 * n * m + 4 * n, flops=2.0 * n * m * d)
    if op == "cp":
        # at least the pairs inside leaves of leaf / 4 points
        return dict(bytes=4 * n * d + 20 * k, flops=3.0 * d * n * case["leaf"] / 8)
    if op == "bnb":
        return dict(bytes=4 * n * d + 20 * k, flops=3.0 * d * (0.0024 * n * (n - 1) + k))
    if op == "serve":
        nq, k = int(24 * nq / math.log(nq)), k // 3
    rows = min(n, nq * k)
    return dict(bytes=4 * nq * d + 16 * nq * k + 4 * rows * d, flops=2.0 * nq * m * d + 3.0 * nq * k * d)


# ---------------------------------------------------- the algorithms in FP64

def _splitmix64(seed, i):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (i.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _r_min(X, beta, k, c):
    """Sec. 5.2: the first radius from 10,000 sampled pair distances (index seed 0)."""
    n, s = X.shape[0], np.arange(10_000)
    i = (_splitmix64(3, 2 * s) % np.uint64(n)).astype(np.int64)
    j = (_splitmix64(3, 2 * s + 1) % np.uint64(n)).astype(np.int64)
    j = np.where(i == j, (j + 1) % n, j)
    v = np.sort((X[i].double() - X[j].double()).norm(dim=1).cpu().numpy())
    rank = math.ceil(min(1.0, (beta * n + k) / n) * len(v) - 1e-9)
    return v[min(max(rank, 1), len(v)) - 1] / c


def _chi_radius(m):
    """t with Pr[chi^2(m) > t^2] = 1/e (Lemma 3), by bisection."""
    a, x = torch.tensor(m / 2.0, dtype=torch.float64), [0.0, 200.0]
    for _ in range(200):
        mid = 0.5 * (x[0] + x[1])
        sf = float(torch.special.gammaincc(a, torch.tensor(mid / 2.0, dtype=torch.float64)))
        x[0 if sf > 1 / math.e else 1] = mid
    return math.sqrt(0.5 * (x[0] + x[1]))


def _nearest(X, x2, q, inside, k):
    """The k nearest rows (FP64 distance, id) among those inside, per query:
    an FP32 ranking with room to spare, then FP64 distances."""
    d2 = (x2 - 2.0 * (q @ X.T) + (q * q).sum(1, keepdim=True)).masked_fill_(~inside, math.inf)
    near = d2.topk(min(X.shape[0], k + 60), dim=1, largest=False)
    ids = near.indices.sort(dim=1).values
    dist = torch.empty(ids.shape, dtype=torch.float64, device=q.device)
    step = max(1, (1 << 26) // (ids.shape[1] * X.shape[1]))
    for a in range(0, len(q), step):
        dist[a:a + step] = (X[ids[a:a + step]].double() - q[a:a + step, None].double()).norm(dim=2)
    dist.masked_fill_(~inside.gather(1, ids), math.inf)
    dist, at = dist.sort(dim=1, stable=True)
    ids = ids.gather(1, at)
    dist, ids = dist[:, :k], ids[:, :k]
    return torch.where(dist.isinf(), -1, ids), dist


def _exact_knn(X, O, x2, Q, A, k, c, beta, r0, t, bc_radius=None):
    """Algorithm 2 (or Algorithm 1 at bc_radius) for every query in FP64."""
    n, dev = X.shape[0], X.device
    budget = math.ceil(beta * n - 1e-9) + k
    qp = Q.double() @ A.double().T
    nq = len(Q)
    ids = torch.full((nq, k), -1, dtype=torch.int64, device=dev)
    dist = torch.full((nq, k), math.inf, dtype=torch.float64, device=dev)
    rounds, rule = np.zeros(nq, np.int32), np.zeros(nq, np.int32)
    ncand, rfin = np.zeros(nq, np.int64), np.zeros(nq)
    step = max(1, min(nq, (1 << 28) // n))
    for a in range(0, nq, step):
        left = torch.arange(a, min(nq, a + step), device=dev)
        r = r0 if bc_radius is None else bc_radius
        while len(left):
            pd = torch.zeros(len(left), n, dtype=torch.float64, device=dev)
            for j in range(O.shape[1]):
                pd.addcmul_(qp[left, j, None] - O[None, :, j], qp[left, j, None] - O[None, :, j])
            pd.sqrt_()
            inside = pd <= t * r
            count = inside.sum(1)
            full = count >= budget
            if bc_radius is None and bool(full.any()):
                rows = full.nonzero()[:, 0]
                cut = pd[rows].topk(budget, dim=1, largest=False).indices
                keep = torch.zeros(len(rows), n, dtype=torch.bool, device=dev)
                keep.scatter_(1, cut, True)
                inside[rows] = keep
            del pd
            i, dd = _nearest(X, x2, Q[left], inside, k)
            del inside
            ids[left], dist[left] = i, dd
            at = left.cpu().numpy()
            rounds[at] += 1
            nxt = c * r
            # rule 1 is tested after r grew; Algorithm 1 tests c r itself
            hit = dd[:, k - 1] <= (c * nxt if bc_radius is None else nxt)
            f, h, cn = full.cpu().numpy(), hit.cpu().numpy(), count.cpu().numpy()
            if bc_radius is not None:
                rule[at] = np.where(f, 2, np.where(h, 1, 0))
                ncand[at] = cn
                none = left[~(full | hit)]
                ids[none], dist[none] = -1, math.inf
                break
            rule[at] = np.where(f, 2, np.where(cn == n, 3, np.where(h, 1, 0)))
            ncand[at] = np.where(f, budget, cn)
            rfin[at] = np.where(f | (cn == n), r, nxt)
            left = left[torch.from_numpy(rule[at] == 0).to(dev)]
            r = nxt
    return ids, dist, dict(rounds=rounds, rule=rule, ncand=ncand, r=rfin)


def _exact_pairs(X, O, k, T):
    """Distances of the k closest of the T pairs nearest in the projection O."""
    n, dev = X.shape[0], X.device
    step = max(1, (1 << 27) // n)
    samp = torch.randint(0, n, (2, 4_000_000), device=dev)
    pd = (O[samp[0]] - O[samp[1]]).norm(dim=1).float()
    cut = float(pd.kthvalue(int(1.2 * T / (n * (n - 1) / 2) * pd.numel())).values)
    got_i, got_j, got_p = [], [], []
    for a in range(0, n, step):
        b = min(n, a + step)
        p = torch.zeros(b - a, n - a, dtype=torch.float64, device=dev)
        for c in range(O.shape[1]):
            t = O[a:b, c, None] - O[None, a:, c]
            p.addcmul_(t, t)
        at = (p <= cut * cut).triu_(1).nonzero()
        got_p.append(p[at[:, 0], at[:, 1]].sqrt())
        got_i.append(at[:, 0] + a)
        got_j.append(at[:, 1] + a)
    keep = torch.cat(got_p).sort(stable=True).indices[:T]
    i, j = torch.cat(got_i)[keep], torch.cat(got_j)[keep]
    dist = torch.empty(len(i), dtype=torch.float64, device=dev)
    step = (1 << 27) // X.shape[1]
    for a in range(0, len(i), step):
        dist[a:a + step] = (X[i[a:a + step]].double() - X[j[a:a + step]].double()).norm(dim=1)
    return dist.sort().values[:k]


def exact(case, seed):
    op = case["op"]
    X, Q, A = _data(case, seed)
    O = X.double() @ A.double().T
    if op == "build":
        return dict(projected=O, perm=None, leaf_off=None, node_lo=None, node_hi=None, node_left=None,
                    node_right=None)
    if op == "cp":
        return None   # which pairs Algorithm 4 meets depends on the leaf hierarchy
    if op == "bnb":
        n = case["n"]
        T = math.ceil(0.0024 * n * (n - 1) - 1e-9) + case["k"]
        return dict(pairs=None, dists=_exact_pairs(X, O, case["k"], T), count=T)
    x2 = (X * X).sum(1)[None]
    t = _chi_radius(case["m"])
    if op == "serve":
        out = []
        for q, k in _requests(case, Q, seed):
            ids, dist, _ = _exact_knn(X, O, x2, torch.from_numpy(q).cuda(), A, k, case["c"], case["beta"],
                                      _r_min(X, case["beta"], k, case["c"]), t)
            out.append((ids, dist))
        return out
    if op == "rcbc":
        ids, dist, st = _exact_knn(X, O, x2, Q, A, 1, case["c"], case["beta"], 0.0, t, bc_radius=case["r"])
        return dict(ids=ids[:, 0], dists=dist[:, 0], stats={f: st[f] for f in ("rule", "ncand", "rounds")})
    ids, dist, st = _exact_knn(X, O, x2, Q, A, case["k"], case["c"], case["beta"],
                               _r_min(X, case["beta"], case["k"], case["c"]), t)
    out = dict(ids=ids, dists=dist, err=(dist.float().double() - dist).abs())
    if case["stats"]:
        out["stats"] = st
    return out
