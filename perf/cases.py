"""Timed cases of the framework: what a user has it do, over the range of
sizes and options it is used at.

Every case goes through the package's public entry points.  Inputs are seeded
graphs with planted clusters (degree-corrected planted partitions: Chung-Lu
weights, power-law cluster sizes, a fraction of clusters built as chains of
parts joined by one or two bridges, so that some of them split), drawn on the
GPU from the seed alone.  The laws are those of the framework's own
configurations.
"""
import math

import numpy as np
import torch

import paper_2509_02590_gb300 as wcc

DEV = "cuda"

# Laws of the input graphs: degree exponent (0 = uniform weights), mean
# degree, largest expected degree (0 = 10 sqrt(n)), cluster-size exponent and
# bounds, share of edges inside clusters, share of chain clusters and the most
# parts of one.
LAWS = {
    # blocks of 50, density 0.2 inside: some are two halves joined by one edge
    "planted": dict(deg_exp=0.0, mean=10.8, deg_max=0, size_exp=1.5, size_min=50, size_max=50,
                    f_in=0.85, chain=0.2, parts=2),
    # communities of 20-2000, mixing 0.3, a tenth of them bridged pairs
    "lfr": dict(deg_exp=2.5, mean=18.4, deg_max=1000, size_exp=1.5, size_min=20, size_max=2000,
                f_in=0.7, chain=0.1, parts=2),
    # clusters of 10-50,000: the largest hold most of the edges
    "broad": dict(deg_exp=2.2, mean=40.0, deg_max=0, size_exp=1.8, size_min=10, size_max=50_000,
                  f_in=0.8, chain=0.05, parts=4),
    # the same graph cut finer: mean cluster size 20
    "fine": dict(deg_exp=2.2, mean=40.0, deg_max=0, size_exp=3.0, size_min=10, size_max=50_000,
                 f_in=0.8, chain=0.05, parts=4),
    # requests of a service: clusters of 20-2000 on graphs of mean degree 20
    "request": dict(deg_exp=2.5, mean=20.0, deg_max=0, size_exp=1.5, size_min=20, size_max=2000,
                    f_in=0.8, chain=0.05, parts=3),
}


def listed():
    return [
        # the smallest call: 1,000 vertices in 20 blocks, graph resident
        dict(name="run_planted_1k", kind="run", law="planted", n=1000, min_size=11, rule="log10"),
        # a small graph from host arrays to host arrays, as in the quick start
        dict(name="host_small", kind="host", law="request", n=1999, min_size=2, rule="log10"),
        # the benchmark's step: CSR from a device edge list, then the refinement
        dict(name="step_lfr_100k", kind="step", law="lfr", n=100_000, min_size=2, rule="log10"),
        # the same graph kept on the device and refined again
        dict(name="run_lfr_100k", kind="run", law="lfr", n=100_000, min_size=2, rule="log10"),
        # a caller that has a CSR: validated copy, then the stricter log2 criterion
        dict(name="csr_log2_33k", kind="csr", law="lfr", n=33_333, min_size=11, rule="log2"),
        # CM: the community step after every cut, at its default resolution
        dict(name="cm_lfr_100k", kind="cm", law="lfr", n=100_000, min_size=2, rule="log10",
             res_den=1000),
        # clusters of up to 50,000 vertices, graph resident
        dict(name="run_broad_1m", kind="run", law="broad", n=1_000_000, min_size=2, rule="log10"),
        # a hundred thousand small clusters, graph resident
        dict(name="run_fine_2m", kind="run", law="fine", n=2_000_003, min_size=2, rule="log10"),
        # loading edges as they come (both directions, repeats and loops among them)
        dict(name="build_raw_1m", kind="build", law="request", n=1_048_583, raw=True),
        # loading a large sorted edge list
        dict(name="build_3m", kind="build", law="broad", n=3_000_000, raw=False),
        # a service: a burst of requests of 10^3 to 10^6 edges, each with its edge list
        dict(name="serve_burst", kind="serve", law="request", requests=48, m_min=1000,
             m_max=1_000_000, min_size=2, rule="log10"),
        # the large configuration: 10M vertices, 200M edges, from the edge list
        dict(name="step_broad_10m", kind="step", law="broad", n=10_000_000, min_size=2,
             rule="log10"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "step", "step", "host", "csr", "cm", "build", "serve"])
    if kind == "serve":
        return dict(kind=kind, law="request", requests=rng.randint(6, 48), m_min=1000,
                    m_max=_log_uniform(rng, 20_000, 1_000_000), min_size=rng.choice([2, 2, 5, 11]),
                    rule="log10")
    if kind == "build":
        raw = rng.random() < 0.5
        return dict(kind=kind, law=rng.choice(["request", "lfr", "broad"]),
                    n=_log_uniform(rng, 1000, 3_000_000), raw=raw)
    if kind == "cm":
        return dict(kind=kind, law=rng.choice(["planted", "lfr", "request"]),
                    n=_log_uniform(rng, 1000, 100_000), min_size=rng.choice([2, 2, 11]),
                    rule="log10", res_den=rng.choice([100, 1000]))
    if kind == "host":
        return dict(kind=kind, law=rng.choice(["planted", "lfr", "request", "fine"]),
                    n=_log_uniform(rng, 1000, 300_000), min_size=rng.choice([2, 2, 11]),
                    rule="log10")
    if kind == "csr":
        return dict(kind=kind, law=rng.choice(["planted", "lfr", "request"]),
                    n=_log_uniform(rng, 1000, 300_000), min_size=rng.choice([2, 11]),
                    rule=rng.choice(["log10", "log2"]))
    return dict(kind=kind, law=rng.choice(["planted", "lfr", "broad", "fine"]),
                n=_log_uniform(rng, 1000, 3_000_000), min_size=rng.choice([2, 2, 5, 11]),
                rule="log10")


# ---- inputs ------------------------------------------------------------------

def _mean_of(expo, lo, hi):
    if abs(expo - 2.0) < 1e-9:
        top = math.log(hi / lo)
    else:
        top = (hi ** (2 - expo) - lo ** (2 - expo)) / (2 - expo)
    return top / ((hi ** (1 - expo) - lo ** (1 - expo)) / (1 - expo))


def _power_law(u, expo, lo, hi):
    a, b = lo ** (1.0 - expo), hi ** (1.0 - expo)
    return (a + u * (b - a)) ** (1.0 / (1.0 - expo))


def _cluster_sizes(rng, n, expo, lo, hi):
    hi = min(hi, n)
    lo = min(lo, hi)
    if lo == hi:
        s = np.full(max(1, n // lo), lo, dtype=np.int64)
    else:
        s = np.zeros(0, dtype=np.int64)
        while s.sum() < n:
            s = np.concatenate([s, np.rint(_power_law(rng.random(1 << 16), expo, lo, hi)).astype(np.int64)])
        s = s[:int(np.searchsorted(np.cumsum(s), n)) + 1]
    s[-1] += n - int(s.sum())
    if s[-1] < 2 and len(s) > 1:  # what is left over joins the cluster before it
        s[-2] += s[-1]
        s = s[:-1]
    return s


def _endpoints(gen, cw, lo, hi):
    """One vertex per entry, in proportion to its weight within [lo, hi)."""
    a, b = cw[lo], cw[hi]
    x = a + torch.rand(a.shape, generator=gen, device=DEV, dtype=torch.float64) * (b - a)
    i = torch.searchsorted(cw, x, right=True) - 1
    return torch.minimum(torch.maximum(i, lo), hi - 1)


def _graph(law, n, m, seed, raw=False):
    """(src, dst, labels) on the GPU: about m undirected edges on n vertices,
    int32; sorted and simple, or with raw as drawn (any order, either
    direction, repeats and loops)."""
    p = LAWS[law]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if p["deg_exp"]:
        top = max(20.0, min(p["deg_max"] or 10 * math.sqrt(n), n / 4))
        mean = 2.0 * m / n
        lo, hi = 0.01, top
        for _ in range(60):
            mid = math.sqrt(lo * hi)
            lo, hi = (mid, hi) if _mean_of(p["deg_exp"], mid, top) < mean else (lo, mid)
        w = _power_law(rng.random(n), p["deg_exp"], lo, top)
    else:
        w = np.ones(n)
    cw_host = np.concatenate([[0.0], np.cumsum(w)])
    # clusters, the edge groups (parts of chains, else whole clusters), bridges
    sizes = _cluster_sizes(rng, n, p["size_exp"], p["size_min"], p["size_max"])
    k = len(sizes)
    starts = np.cumsum(sizes) - sizes
    parts = rng.integers(2, p["parts"] + 1, size=k)
    parts = np.where((rng.random(k) < p["chain"]) & (sizes >= 6 * parts), parts, 1)
    first = np.cumsum(parts) - parts
    owner = np.repeat(np.arange(k), parts)
    at = np.arange(len(owner)) - first[owner]
    length = sizes[owner] // parts[owner]
    g_lo = starts[owner] + at * length
    g_hi = np.where(at == parts[owner] - 1, starts[owner] + sizes[owner], g_lo + length)
    joint = np.nonzero(at < parts[owner] - 1)[0]
    joint = np.repeat(joint, rng.integers(1, 3, size=len(joint)))
    bu = g_lo[joint] + (rng.random(len(joint)) * (g_hi - g_lo)[joint]).astype(np.int64)
    bv = g_lo[joint + 1] + (rng.random(len(joint)) * (g_hi - g_lo)[joint + 1]).astype(np.int64)
    gw = cw_host[g_hi] - cw_host[g_lo]
    glen = (g_hi - g_lo).astype(np.float64)
    m_g = np.minimum(np.rint(1.15 * p["f_in"] * m * gw / gw.sum()),
                     np.floor(0.25 * glen * (glen - 1))).astype(np.int64)
    cw = torch.from_numpy(cw_host).to(DEV)
    lo_t, hi_t = torch.from_numpy(g_lo).to(DEV), torch.from_numpy(g_hi).to(DEV)
    us, vs = [torch.from_numpy(bu).to(DEV)], [torch.from_numpy(bv).to(DEV)]
    # inside the groups, in slices that bound the memory of the draw
    ends = np.cumsum(m_g)
    g0 = 0
    while g0 < len(m_g):
        g1 = max(g0 + 1, int(np.searchsorted(ends, (ends[g0 - 1] if g0 else 0) + (1 << 26))))
        rep = torch.repeat_interleave(torch.arange(g0, g1, device=DEV),
                                      torch.from_numpy(m_g[g0:g1]).to(DEV))
        us.append(_endpoints(gen, cw, lo_t[rep], hi_t[rep]))
        vs.append(_endpoints(gen, cw, lo_t[rep], hi_t[rep]))
        g0 = g1
    # between the clusters, over the whole graph
    cluster = torch.repeat_interleave(torch.arange(k, device=DEV), torch.from_numpy(sizes).to(DEV))
    left = max(0, m - int(m_g.sum() / 1.15))
    zero, top_id = torch.zeros((), dtype=torch.long, device=DEV), torch.full((), n, dtype=torch.long, device=DEV)
    while left > 0:
        c = min(left, 1 << 26)
        u = _endpoints(gen, cw, zero.expand(c), top_id.expand(c))
        v = _endpoints(gen, cw, zero.expand(c), top_id.expand(c))
        keep = cluster[u] != cluster[v]
        us.append(u[keep])
        vs.append(v[keep])
        left -= c
    del cw
    # vertices and label values in random order
    perm = torch.randperm(n, generator=gen, device=DEV)
    value = torch.randperm(3 * k, generator=gen, device=DEV)[:k]
    labels = torch.empty(n, dtype=torch.int32, device=DEV)
    labels[perm] = value[cluster].int()
    u, v = perm[torch.cat(us)], perm[torch.cat(vs)]
    del us, vs, perm, cluster
    if raw:
        mix = torch.randperm(u.numel(), generator=gen, device=DEV)
        flip = torch.rand(u.numel(), generator=gen, device=DEV) < 0.5
        u, v = u[mix], v[mix]
        return torch.where(flip, v, u).int(), torch.where(flip, u, v).int(), labels
    key = torch.minimum(u, v) * n + torch.maximum(u, v)
    key = torch.unique(key[u != v])
    return (key // n).int(), (key % n).int(), labels


def _edges(case):
    """Undirected edges asked for: the law's mean degree."""
    return int(case["n"] * LAWS[case["law"]]["mean"] / 2)


def _request_sizes(case):
    """Edge counts spread evenly over the logarithm of their range, in one
    mixed order."""
    r, a, b = case["requests"], case["m_min"], case["m_max"]
    m = a * (b / a) ** ((np.arange(r) + 0.5) / r)
    return [int(x) for x in np.random.default_rng(r).permutation(np.rint(m))]


def prepare(case, seed):
    s = dict(case=case)
    if case["kind"] == "serve":
        s["requests"] = []
        for i, m in enumerate(_request_sizes(case)):
            n = max(100, m // 10)
            src, dst, lab = _graph(case["law"], n, m, 1000 * seed + i)
            s["requests"].append((src.cpu().pin_memory(), dst.cpu().pin_memory(), n,
                                  lab.cpu().numpy()))
        return s
    n = case["n"]
    src, dst, lab = _graph(case["law"], n, _edges(case), seed, raw=case.get("raw", False))
    if case["kind"] == "host":
        s["src"], s["dst"], s["labels"] = src.cpu().numpy(), dst.cpu().numpy(), lab.cpu().numpy()
    elif case["kind"] == "step":
        s["src"], s["dst"], s["labels"] = src, dst, lab
    elif case["kind"] == "build":
        # the caller's own buffers for the CSR, with room for every entry
        m = _edges(case)
        s["src"], s["dst"] = src[:m], dst[:m]
        s["off"] = torch.empty(n + 1, dtype=torch.int64, device=DEV)
        s["adj"] = torch.full((2 * m,), -1, dtype=torch.int32, device=DEV)
    else:
        s["labels"] = lab
        s["graph"] = wcc.WccGraph.from_edges(src, dst, n)
        if case["kind"] == "csr":
            s["off"], s["adj"] = s["graph"].csr(device=True)
            s.pop("graph").close()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        with wcc.WccServer(8 << 30) as server:
            tickets = [server.submit_edges(src, dst, n, lab, min_size=case["min_size"],
                                           rule=case["rule"])
                       for src, dst, n, lab in state["requests"]]
            return [server.wait(t)[0] for t in tickets]
    if kind == "run":
        return state["graph"].run(state["labels"], min_size=case["min_size"], rule=case["rule"])
    if kind == "cm":
        return state["graph"].run_cm(state["labels"], (1, case["res_den"]),
                                     min_size=case["min_size"], rule=case["rule"])
    if kind == "csr":
        with wcc.WccGraph.from_csr(state["off"], state["adj"]) as g:
            return g.run(state["labels"], min_size=case["min_size"], rule=case["rule"])
    with wcc.WccGraph.from_edges(state["src"], state["dst"], case["n"]) as g:
        if kind == "build":
            wcc.wcc_graph_export_csr(g.handle, state["off"].data_ptr(), state["adj"].data_ptr(), 1,
                                     torch.cuda.current_stream().cuda_stream)
            return state["off"], state["adj"]
        return g.run(state["labels"], min_size=case["min_size"], rule=case["rule"])


def work(case):
    """Bytes of one pass: a refinement reads the labels, the row offsets and
    every adjacency entry and writes labels; a build reads the edges and
    writes offsets and columns; loading a CSR reads and writes it.  The
    operations are one comparison per adjacency entry."""
    kind = case["kind"]
    if kind == "serve":
        # the mean of the log-uniform edge counts
        a, b = case["m_min"], case["m_max"]
        m = case["requests"] * (b - a) / math.log(b / a)
        n = m / 10
    else:
        n, m = case["n"], _edges(case)
    csr, refine, build = 8 * n + 8 * m, 8 * n + 8 * n + 8 * m, 8 * m + 8 * n + 8 * m
    total = {"run": refine, "cm": refine, "csr": 2 * csr + refine, "build": build,
             "step": build + refine, "host": build + refine, "serve": build + refine}[kind]
    return {"bytes": float(total), "flops": float(2 * m)}


def exact(case, seed):
    """Every output is a whole number: there is nothing to be off from."""
    return None
