"""The calls whose time is measured: what a user of this library has it do.

Every case is one pass through the package's public entry points on seeded
synthetic inputs: planted-partition graphs (equal communities and Poisson
degrees, or power-law communities and degrees) and Gaussian-mixture kNN graphs,
with input partitions that merge, split and locally relabel the planted one.
A case is a dict of plain values:

* ``call``   what a pass does (see ``run``)
* ``graph``  ``sbm``, ``lfr`` or ``knn``;  ``n`` vertices, ``k`` input partitions
* ``deg``    mean degree (sbm, lfr);  ``mu`` share of edges that leave a community
* ``jobs``, ``nmin``, ``nmax``, ``kmin``, ``kmax``  the mix of a batch or a request stream
* ``active_set``, ``empty_moves``, ``colour_batched``  the library's options of these names
"""
import math

import numpy as np
import torch

import paper_2408_11331_gb300 as cc

DEV = "cuda"
COMPONENTS, DIM, NEIGHBOURS = 200, 50, 15  # of the kNN graphs


def listed():
    return [
        # The smallest call: one small graph already on the device, solved
        # again and again (a parameter scan, a consensus inside another
        # method).  Its time is launches, gaps and the host's waits.
        dict(name="sbm_small", call="resident", graph="sbm", n=1000, k=10, deg=14.0, mu=0.3),
        # One modest job from host arrays to host labels: load, solve, read
        # the result, release.  The common interactive use.
        dict(name="lfr_call_host", call="host", graph="lfr", n=20011, k=12, deg=20.0, mu=0.3),
        # A large job whose inputs are already in device buffers (made by
        # another GPU program), from those buffers to host labels.
        dict(name="lfr_call_dev", call="device", graph="lfr", n=1000000, k=20, deg=20.0, mu=0.3),
        # The power-law benchmark job, resident inputs.
        dict(name="lfr_large", call="resident", graph="lfr", n=1000000, k=20, deg=20.0, mu=0.3),
        # Mid-size job with an odd n and a k that fills no quad of partitions,
        # with the option that re-scores only what changed.
        dict(name="lfr_ragged_active", call="resident", graph="lfr", n=150001, k=37, deg=15.0, mu=0.45, active_set=1),
        # The single-cell shaped job, the largest that is solved: resident inputs.
        dict(name="knn_large", call="resident", graph="knn", n=2000000, k=50),
        # A day's worth of small jobs solved together: create the batch, run
        # it, read all labels and objectives.
        dict(name="batch_mix", call="batch", graph="mix", jobs=48, nmin=200, nmax=40000, kmin=5, kmax=64, active_set=1),
        # Requests that arrive faster than they are served, through the
        # request loop: submit all, drain, collect every result.
        dict(name="serve_mix", call="serve", graph="lfr", jobs=40, nmin=1000, nmax=100000, kmin=8, kmax=32, active_set=1),
        # Refining a given consensus (a resumed run, an update after a change
        # of the inputs), where a vertex may also leave for a cluster of its own.
        dict(name="warm_refine", call="warm", graph="lfr", n=300007, k=24, deg=20.0, mu=0.3, empty_moves=1),
        # The better-quality schedule, one colour class at a time.
        dict(name="colour_mid", call="resident", graph="lfr", n=100000, k=8, deg=20.0, mu=0.3, colour_batched=1),
        # Distances of a consensus to its input partitions (evaluation).
        dict(name="metrics_large", call="metrics", graph="knn", n=1000000, k=50),
        # All distances between the input partitions (grouping them before
        # the consensus).
        dict(name="distances_mid", call="distances", graph="lfr", n=200003, k=24, deg=20.0, mu=0.3),
    ]


def _log_int(rng, lo, hi):
    """An integer, log-uniform on [lo, hi]; three in four of them as drawn, so mostly odd sizes."""
    x = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, x if rng.random() < 0.75 else x // 100 * 100))


def draw(rng):
    what = rng.choice(("resident", "resident", "knn", "host", "device", "batch", "serve", "warm", "colour",
                       "metrics", "distances"))
    kind = rng.choice(("lfr", "lfr", "sbm"))
    deg, mu = round(rng.uniform(10, 30), 2), round(rng.uniform(0.1, 0.5), 3)
    if what == "resident":
        return dict(call="resident", graph=kind, n=_log_int(rng, 1000, 1000000), k=rng.randint(5, 40), deg=deg, mu=mu,
                    active_set=rng.randint(0, 1))
    if what == "knn":
        return dict(call="resident", graph="knn", n=_log_int(rng, 20000, 1500000), k=rng.randint(8, 50))
    if what == "host":
        return dict(call="host", graph=kind, n=_log_int(rng, 1000, 200000), k=rng.randint(5, 40), deg=deg, mu=mu)
    if what == "device":
        return dict(call="device", graph=kind, n=_log_int(rng, 10000, 1000000), k=rng.randint(5, 40), deg=deg, mu=mu)
    if what == "batch":
        return dict(call="batch", graph="mix", jobs=_log_int(rng, 4, 64), nmin=200, nmax=_log_int(rng, 2000, 40000),
                    kmin=5, kmax=rng.randint(10, 64), active_set=1)
    if what == "serve":
        return dict(call="serve", graph="lfr", jobs=_log_int(rng, 4, 40), nmin=1000, nmax=_log_int(rng, 10000, 100000),
                    kmin=8, kmax=rng.randint(10, 32), active_set=1)
    if what == "warm":
        return dict(call="warm", graph=kind, n=_log_int(rng, 2000, 500000), k=rng.randint(5, 40), deg=deg, mu=mu,
                    empty_moves=rng.randint(0, 1))
    if what == "colour":
        return dict(call="resident", graph=kind, n=_log_int(rng, 2000, 200000), k=rng.randint(5, 20), deg=deg, mu=mu,
                    colour_batched=1)
    if what == "metrics":
        return dict(call="metrics", graph=rng.choice(("lfr", "knn")), n=_log_int(rng, 20000, 1000000),
                    k=rng.randint(5, 50), deg=deg, mu=mu)
    return dict(call="distances", graph=kind, n=_log_int(rng, 2000, 300000), k=rng.randint(5, 24), deg=deg, mu=mu)


# ---- inputs (made on the GPU; every draw from the seed's own generators) ----

class _Gen:
    def __init__(self, seed):
        self.dev = torch.Generator(device=DEV)
        self.dev.manual_seed(seed)
        self.host = np.random.default_rng(seed)

    def rand(self, *shape):
        return torch.rand(shape, generator=self.dev, device=DEV)

    def perm(self, n):
        return torch.randperm(n, generator=self.dev, device=DEV)

    def below(self, hi, n):
        return torch.randint(0, hi, (n,), generator=self.dev, device=DEV)


def _power_law(u, expo, lo, hi):
    a = 1.0 - expo
    return (lo ** a + u * (hi ** a - lo ** a)) ** (1.0 / a)


def _community_sizes(g, n, kind):
    """SBM: communities of 20 to 500 vertices; LFR-style: power law 1.5 on [50, 5000]."""
    lo, hi = (20, 500) if kind == "sbm" else (min(50, n), min(5000, n))
    count = max(16, int(8 * n / (lo + hi)) + 16)
    u = g.host.random(count)
    s = np.rint(lo + u * (hi - lo)) if kind == "sbm" else np.rint(_power_law(u, 1.5, lo, hi))
    while s.sum() < n:
        s = np.concatenate([s, s])
    ends = np.minimum(np.cumsum(s.astype(np.int64)), n)
    sizes = np.diff(np.concatenate([[0], ends]))
    return sizes[sizes > 0]


def _csr(n, u, v):
    """Undirected pairs -> symmetric CSR with sorted rows, no repeats, no self-loops."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique_consecutive(torch.sort(torch.cat([u * n + v, v * n + u])).values)
    rows = torch.div(key, n, rounding_mode="floor")
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return off, (key - rows * n).to(torch.int32)


def _planted(g, kind, n, deg, mu):
    """Configuration-model graph with planted communities: (off, col, truth)."""
    sizes = torch.from_numpy(_community_sizes(g, n, kind)).to(DEV)
    truth = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), sizes)
    if kind == "sbm":
        d = torch.poisson(torch.full((n,), float(deg), device=DEV), generator=g.dev).to(torch.int64)
    else:
        truth = truth[g.perm(n)]
        hi = float(min(1000, max(n // 10, int(2 * deg))))
        lo_d, hi_d = 1.0, hi
        for _ in range(60):  # the lower cut-off that gives the mean degree
            mid = 0.5 * (lo_d + hi_d)
            a, b = -1.5, -0.5
            mean = (a / b) * (hi ** b - mid ** b) / (hi ** a - mid ** a)
            lo_d, hi_d = (mid, hi_d) if mean < deg else (lo_d, mid)
        d = torch.round(_power_law(g.rand(n).double(), 2.5, lo_d, hi)).to(torch.int64)
    inside = torch.minimum(torch.round((1.0 - mu) * d).to(torch.int64), sizes[truth] - 1)
    ids = torch.arange(n, device=DEV)
    # stubs inside: shuffled, then grouped by community, and paired in order
    stub = torch.repeat_interleave(ids, inside)
    stub = stub[g.perm(len(stub))]
    stub = stub[torch.sort(truth[stub], stable=True).indices]
    stub = stub[: len(stub) // 2 * 2].view(-1, 2)
    same = truth[stub[:, 0]] == truth[stub[:, 1]]
    out = torch.repeat_interleave(ids, d - inside)
    out = out[g.perm(len(out))]
    out = out[: len(out) // 2 * 2].view(-1, 2)
    cross = truth[out[:, 0]] != truth[out[:, 1]]
    pairs = torch.cat([stub[same], out[cross]])
    off, col = _csr(n, pairs[:, 0], pairs[:, 1])
    return off, col, truth


def _relabel(g, lab, off, col, rho):
    """With probability rho a vertex takes the label of a random neighbour."""
    n = len(lab)
    deg = off[1:] - off[:-1]
    pick = (g.rand(n) < rho) & (deg > 0)
    at = off[:-1] + torch.minimum((g.rand(n).double() * deg).to(torch.int64), (deg - 1).clamp(min=0))
    at = torch.where(pick, at, torch.zeros_like(at))
    return torch.where(pick, lab[col[at].long()], lab) if len(col) else lab


def _perturbed(g, truth, off, col, k, rho_hi):
    """k input partitions: planted communities merged, split and relabelled."""
    K = int(truth.max()) + 1
    labels = torch.empty((k, len(truth)), dtype=torch.int32, device=DEV)
    for i in range(k):
        merge = g.host.random(K) < 0.2
        root = np.arange(K)
        root[merge] = np.floor(g.host.random(K) * np.arange(K)).astype(np.int64)[merge]  # some smaller id
        for _ in range(max(1, K.bit_length())):
            root = root[root]
        split = g.host.random(K) < 0.2
        lab = torch.from_numpy(root).to(DEV)[truth]
        half = torch.from_numpy(split).to(DEV)[truth] & (g.rand(len(truth)) < 0.5)
        lab = torch.where(half, K + truth, lab)
        labels[i] = _relabel(g, lab, off, col, g.host.uniform(0.05, rho_hi)).to(torch.int32)
    return labels


def _knn(g, n, k):
    """Symmetrised kNN graph of a Gaussian mixture (neighbours inside each
    component, exact) and k partitions of 50 to 2000 clusters: components
    grouped at random, or cut by rank along a random direction; 10% relabelled."""
    comps = min(COMPONENTS, max(2, n // 100))
    w = g.host.dirichlet(np.ones(comps))
    sizes = np.maximum(g.host.multinomial(n, w), 0)
    truth = torch.repeat_interleave(torch.arange(comps, device=DEV), torch.from_numpy(sizes).to(DEV))
    x = torch.randn(n, DIM, generator=g.dev, device=DEV)
    x *= torch.from_numpy(g.host.uniform(0.5, 2.0, comps)).float().to(DEV)[truth][:, None]
    sq = (x * x).sum(1)
    ends = np.concatenate([[0], np.cumsum(sizes)])
    us, vs = [], []
    for c in range(comps):
        lo, hi = int(ends[c]), int(ends[c + 1])
        m = min(NEIGHBOURS, hi - lo - 1)
        if m < 1:
            continue
        for s in range(lo, hi, 8192):
            e = min(hi, s + 8192)
            d = torch.addmm(sq[None, lo:hi], x[s:e], x[lo:hi].T, beta=1.0, alpha=-2.0)
            d[torch.arange(e - s, device=DEV), torch.arange(s - lo, e - lo, device=DEV)] = float("inf")
            vs.append((torch.topk(d, m, dim=1, largest=False).indices + lo).reshape(-1))
            us.append(torch.repeat_interleave(torch.arange(s, e, device=DEV), m))
    where = g.perm(n)  # vertex ids have nothing to do with the components
    off, col = _csr(n, where[torch.cat(us)], where[torch.cat(vs)])
    del us, vs
    truth_v = torch.empty_like(truth)
    truth_v[where] = truth
    labels = torch.empty((k, n), dtype=torch.int32, device=DEV)
    start = torch.from_numpy(ends).to(DEV)
    size_t = torch.from_numpy(sizes).to(DEV)
    for i in range(k):
        K = int(np.rint(np.exp(g.host.uniform(math.log(50), math.log(2000)))))
        if K <= comps:
            group = torch.from_numpy(np.concatenate([np.arange(K), g.host.integers(0, K, comps - K)])).to(DEV)
            lab = group[torch.from_numpy(g.host.permutation(comps)).to(DEV)][truth]
        else:
            q = -(-K // comps)
            proj = x @ torch.from_numpy(g.host.standard_normal(DIM)).float().to(DEV)
            by = torch.sort(proj).indices
            by = by[torch.sort(truth[by], stable=True).indices]  # component by component, by rank
            rank = torch.empty(n, dtype=torch.int64, device=DEV)
            rank[by] = torch.arange(n, device=DEV)
            rank -= start[truth]
            lab = truth * q + torch.div(rank * q, size_t[truth], rounding_mode="floor")
        placed = torch.empty_like(lab)
        placed[where] = lab
        labels[i] = _relabel(g, placed, off, col, 0.1).to(torch.int32)
    return off, col, truth_v, labels


def _job(g, kind, n, k, deg, mu):
    if kind == "knn":
        return _knn(g, n, k)
    off, col, truth = _planted(g, kind, n, deg, mu)
    return off, col, truth, _perturbed(g, truth, off, col, k, 0.3 if kind == "sbm" else 0.4)


def _mix(case):
    """(kind, n, k, deg, mu) of each job of a batch or request stream: n
    log-uniform (one job per stratum) in random order.  The sizes follow from
    the case; the graphs and partitions from the seed."""
    rng = np.random.default_rng([case[f] for f in ("jobs", "nmin", "nmax", "kmin", "kmax")])
    jobs = case["jobs"]
    q = rng.permutation((np.arange(jobs) + rng.random(jobs)) / jobs)
    ns = np.rint(case["nmin"] * (case["nmax"] / case["nmin"]) ** q).astype(int)
    kinds = ["sbm" if case["graph"] == "mix" and j % 2 == 0 else "lfr" for j in range(jobs)]
    return [(kinds[j], int(ns[j]), int(rng.integers(case["kmin"], case["kmax"] + 1)), float(rng.uniform(10, 30)),
             float(rng.uniform(0.1, 0.5))) for j in range(jobs)]


def _first_ids(lab):
    """Cluster ids as the library names them: each cluster by its least vertex."""
    n = len(lab)
    order = torch.sort(lab, stable=True).indices
    s = lab[order]
    head = torch.ones(n, dtype=torch.bool, device=DEV)
    head[1:] = s[1:] != s[:-1]
    first = order[head][torch.cumsum(head.to(torch.int64), 0) - 1]
    out = torch.empty_like(first)
    out[order] = first
    return out.to(torch.int32)


def _inputs(case, seed):
    return _job(_Gen(seed), case["graph"], case["n"], case["k"], case.get("deg", 0.0), case.get("mu", 0.0))


def _host(off, col, labels):
    return off.cpu().numpy(), col.cpu().numpy(), labels.cpu().numpy()


def _options(case):
    o = cc.cc_default_options()
    for f in ("active_set", "empty_moves", "colour_batched"):
        setattr(o, f, int(case.get(f, 0)))
    return o


def _resident(case, off, col, labels):
    torch.cuda.synchronize()  # the inputs are read on the library's own stream
    return cc.Consensus.from_device(case["n"], len(col), off.data_ptr(), col.data_ptr(), case["k"], labels.data_ptr(),
                                    _options(case))


def prepare(case, seed):
    call = case["call"]
    if call in ("batch", "serve"):
        g, jobs = _Gen(seed), []
        for kind, n, k, deg, mu in _mix(case):
            off, col, _, labels = _job(g, kind, n, k, deg, mu)
            jobs.append(_host(off, col, labels))
        s = dict(call=call, jobs=jobs, options=_options(case))
        if call == "serve":
            s["server"] = cc.Server(options=_options(case))
        return s
    off, col, truth, labels = _inputs(case, seed)
    if call == "host":
        return dict(call=call, arrays=_host(off, col, labels), options=_options(case))
    if call == "device":
        torch.cuda.synchronize()
        return dict(call=call, off=off, col=col, labels=labels, n=case["n"], k=case["k"], options=_options(case))
    s = dict(call=call, job=_resident(case, off, col, labels))
    if call == "warm":
        s["start"] = _first_ids(labels[0]).cpu().numpy()
    if call == "metrics":
        s["job"].set_cluster_ids(_first_ids(truth).cpu().numpy())
    return s


def _solve(job):
    sweeps = job.run_until_converged()
    return {"labels": job.consensus_labels(), "F": job.objective(), "sweeps": sweeps}


def run(s):
    call = s["call"]
    if call == "resident":  # the job from its singleton start to its labels
        s["job"].reset()
        return _solve(s["job"])
    if call == "warm":  # the same from a given consensus
        s["job"].set_cluster_ids(s["start"])
        return _solve(s["job"])
    if call == "host":  # from host arrays to host labels
        with cc.Consensus(*s["arrays"], s["options"]) as job:
            return _solve(job)
    if call == "device":  # from device buffers to host labels
        with cc.Consensus.from_device(s["n"], len(s["col"]), s["off"].data_ptr(), s["col"].data_ptr(), s["k"],
                                      s["labels"].data_ptr(), s["options"]) as job:
            return _solve(job)
    if call == "batch":
        with cc.ConsensusBatch(s["jobs"], s["options"]) as batch:
            batch.run_until_converged()
            return {"labels": batch.consensus_labels(), "F": np.array([batch.objective(j) for j in range(batch.jobs)])}
    if call == "serve":
        srv = s["server"]
        tickets = [srv.submit(*job) for job in s["jobs"]]
        srv.drain()
        got = [srv.result(t, pop=True) for t in tickets]
        return {"labels": np.concatenate([r["labels"] for r in got]), "F": np.array([r["F"] for r in got]),
                "sweeps": np.array([r["sweeps"] for r in got])}
    if call == "metrics":
        return s["job"].metrics()
    return s["job"].partition_distances()


def work(case):
    """Bytes: each graph and label array read once, each result written once.
    The method is integer counting: no floating-point operations to speak of."""
    call = case["call"]
    if call in ("batch", "serve"):
        ratio = case["nmax"] / case["nmin"]
        n = case["jobs"] * (case["nmax"] - case["nmin"]) / math.log(ratio)  # mean of a log-uniform n
        return {"bytes": n * (8 + 4 * 20 + 4 * 0.5 * (case["kmin"] + case["kmax"]) + 4), "flops": 0}
    n, k = case["n"], case["k"]
    if call == "metrics":
        return {"bytes": 4 * n * (k + 1) + 32 * k, "flops": 0}
    if call == "distances":
        return {"bytes": 4 * n * k + 32 * k * k, "flops": 0}
    nnz = n * (26 if case["graph"] == "knn" else case["deg"])
    return {"bytes": 8 * (n + 1) + 4 * nnz + 4 * n * k + 4 * n + (4 * n if call == "warm" else 0), "flops": 0}


# ---- the distances in 64 bits, from the definitions ------------------------

def _distances(a, b):
    """(Mirkin, split-join, Rand distance, variation of information) of two labelings."""
    n = len(a)
    _, a = torch.unique(a, return_inverse=True)
    _, b = torch.unique(b, return_inverse=True)
    nb = int(b.max()) + 1
    pair, cnt = torch.unique(a * nb + b, return_counts=True)
    ca, cb = torch.bincount(a), torch.bincount(b)
    mirkin = int((ca * ca).sum() + (cb * cb).sum() - 2 * (cnt * cnt).sum())
    ra, rb = torch.div(pair, nb, rounding_mode="floor"), pair % nb
    top_a = torch.zeros_like(ca).scatter_reduce_(0, ra, cnt, "amax")
    top_b = torch.zeros_like(cb).scatter_reduce_(0, rb, cnt, "amax")
    p = cnt.double() / n
    pa, pb = ca.double()[ra] / n, cb.double()[rb] / n
    vi = float(-(p * (torch.log(p / pa) + torch.log(p / pb))).sum())
    return mirkin, 2 * n - int(top_a.sum()) - int(top_b.sum()), mirkin / (n * (n - 1.0)), vi


def exact(case, seed):
    if case["call"] not in ("metrics", "distances"):
        return None  # whole numbers: the consensus and its objective
    _, _, truth, labels = _inputs(case, seed)
    k = case["k"]
    if case["call"] == "metrics":
        d, shape = [_distances(truth, labels[i]) for i in range(k)], (k,)
    else:
        d, shape = [_distances(labels[i], labels[j]) for i in range(k) for j in range(k)], (k, k)
    out = {}
    for t, f in enumerate(("mirkin", "split_join", "rand_distance", "vi")):
        out[f] = np.array([r[t] for r in d], dtype=np.int64 if t < 2 else np.float64).reshape(shape)
    return out
