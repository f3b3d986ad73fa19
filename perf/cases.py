"""The library's work as its users have it done: timed cases over the public entry points.

Each case names a kind of call and the graph (or feature rows) that it runs on.  Graphs are random, built on the GPU
from the seed: Erdos-Renyi, R-MAT, Barabasi-Albert, power-law configuration model and batches of Watts-Strogatz
graphs, at the sizes of this repository's standard workloads and down to the smallest that callers send.

  listed()            the cases that are always timed
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs, context and output buffers that a program holds before the call
  run(state)          one pass through the public entry point
  work(case)          bytes and operations that a pass cannot do without
  exact(case, seed)   the floating outputs in 64 bits, by plain torch
"""
import math

import torch

import paper_2306_00606_gb300 as ef

OUT_TYPES = {"ef": torch.float64, "n_clusters": torch.int64, "s": torch.int64, "t": torch.float64,
             "triangles": torch.int64, "flag": torch.uint8}


# ------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest calls: EF of one contact network of a few thousand people, default options.  Launches and
        # the host's part of the call count.
        {"name": "er_2k_fp64", "kind": "compute", "graph": "er", "n": 2000, "degree": 8, "precision": "fp64",
         "replay": False, "outputs": "ef"},
        # Repeated calls on a small graph with hubs, as a sweep over networks or a monitoring loop makes them:
        # validation on the device, the call replayed as a CUDA graph.
        {"name": "rmat_64k_fp32c_replay", "kind": "compute", "graph": "rmat", "n": 65536, "degree": 16,
         "precision": "fp32c", "replay": True, "outputs": "ef"},
        # An ordinary large graph with the default precision and every per-node output.
        {"name": "ba_1m_fp64_all", "kind": "compute", "graph": "ba", "n": 1_000_000, "degree": 10,
         "precision": "fp64", "replay": False, "outputs": "ef,n_clusters,s,t,triangles,flag"},
        # The headline: a social-network-sized graph with heavy hubs, repeated calls.
        {"name": "plcm_4m_fp32c_replay", "kind": "compute", "graph": "plcm", "n": 4_000_000, "degree": 3,
         "precision": "fp32c", "replay": True, "outputs": "ef"},
        # The largest exact call in full precision: the same family at minimum degree 6 (about 8.7e7 entries).
        {"name": "plcm_4m_min6_fp64", "kind": "compute", "graph": "plcm", "n": 4_000_000, "degree": 6,
         "precision": "fp64", "replay": False, "outputs": "ef"},
        # A graph that arrives in host memory and whose EF goes back there (the call copies both ways).
        {"name": "plcm_1m_fp64_host", "kind": "host", "graph": "plcm", "n": 1_000_003, "degree": 3,
         "precision": "fp64"},
        # Thousands of uneven small-world graphs in one call (an ensemble study).
        {"name": "ws_4096_fp32c", "kind": "batch", "graph": "ws", "n": 4096, "degree": 12, "precision": "fp32c"},
        # Exact EF of a watch list only.
        {"name": "nodes_2k_of_ba_1m_fp64", "kind": "nodes", "graph": "ba", "n": 1_000_000, "degree": 10,
         "precision": "fp64", "k": 2000},
        # Epidemic simulations that check EF against outbreaks: sizes, lengths, peaks and spreading power.
        {"name": "sir_512_on_ba_500k", "kind": "sir", "graph": "ba", "n": 500_000, "degree": 10, "k": 512},
        # Scoring the feature rows of a large graph with the trained network.
        {"name": "mlp_forward_8m", "kind": "forward", "n": 8_000_001},
        # Loss and gradient of the network over a training set.
        {"name": "mlp_grad_1m", "kind": "grad", "n": 1_000_000},
        # Ranking all nodes of a very large graph: features, network, selection, exact EF of the candidates.
        {"name": "rank_ba_16m_fp64", "kind": "rank", "graph": "ba", "n": 16_000_000, "degree": 8,
         "precision": "fp64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compute", "compute", "compute", "compute", "host", "batch", "nodes", "sir", "forward", "grad",
                       "rank"])
    if kind == "forward":
        return {"kind": kind, "n": _log_int(rng, 500, 8_000_000)}
    if kind == "grad":
        return {"kind": kind, "n": _log_int(rng, 500, 1_000_000)}
    c = {"kind": kind}
    if kind == "batch":
        c.update(graph="ws", n=_log_int(rng, 4, 4096), degree=12)
    elif kind == "sir":
        c.update(graph=rng.choice(["ba", "er"]), n=_log_int(rng, 2000, 500_000), degree=rng.choice([6, 8, 10]),
                 k=_log_int(rng, 20, 512))
        return c
    elif kind in ("nodes", "rank"):
        c.update(graph="ba", n=_log_int(rng, 20_000, 1_000_000 if kind == "nodes" else 16_000_000),
                 degree=rng.choice([6, 8]))
        if kind == "nodes":
            c["k"] = _log_int(rng, 100, 20_000)
    else:
        c["graph"] = rng.choice(["er", "rmat", "ba", "plcm"])
        if c["graph"] == "rmat":
            c.update(n=1 << rng.randint(10, 18), degree=rng.choice([4, 8, 16, 32]))
        elif c["graph"] == "plcm":
            c.update(n=_log_int(rng, 2000, 2_000_000 if kind == "host" else 4_000_000), degree=rng.randint(2, 6))
        else:
            c.update(n=_log_int(rng, 500, 1_000_000 if kind == "host" else 4_000_000), degree=rng.choice([4, 8, 10, 14]))
    c["precision"] = "fp64" if kind == "rank" else rng.choice(["fp64", "fp32c"])
    if kind == "compute":
        c["replay"] = rng.random() < 0.5
        c["outputs"] = rng.choice(["ef", "ef,n_clusters,s,t,triangles,flag"])
    return c


# ------------------------------------------------------------------ graphs

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(0x5EED0000 + seed)
    return g


def _csr(n, u, v):
    """Symmetric sorted simple CSR (int32) from undirected pairs; loops dropped, repeated pairs merged."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    rows = torch.div(key, n, rounding_mode="floor")
    col = (key - rows * n).to(torch.int32)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rp.to(torch.int32), col


def _erdos_renyi(g, n, degree):
    e = n * degree // 2
    u = torch.randint(n, (e,), generator=g, device="cuda")
    v = torch.randint(n, (e,), generator=g, device="cuda")
    return _csr(n, u, v)


def _rmat(g, n, degree):
    """R-MAT with the Graph500 probabilities (0.57, 0.19, 0.19, 0.05); n a power of two."""
    e = n * degree // 2
    u = torch.zeros(e, dtype=torch.int64, device="cuda")
    v = torch.zeros(e, dtype=torch.int64, device="cuda")
    for _ in range(n.bit_length() - 1):
        r = torch.rand(e, generator=g, device="cuda")
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return _csr(n, u, v)


def _barabasi_albert(g, n, degree):
    """Preferential attachment: edge e joins node e // m to an end of an earlier edge, drawn uniformly."""
    m = degree // 2
    e = n * m
    k = torch.arange(e, dtype=torch.int64, device="cuda")
    end = (torch.rand(e, generator=g, device="cuda", dtype=torch.float64) * (2 * k + 1)).to(torch.int64)
    drawn = end.clone()          # end 2e is edge e's own node, end 2e + 1 its target (the end that it drew)
    while True:
        odd = torch.nonzero(end & 1).squeeze(1)
        if odd.numel() == 0:
            break
        end[odd] = drawn[torch.div(end[odd] - 1, 2, rounding_mode="floor")]
    return _csr(n, torch.div(k, m, rounding_mode="floor"), torch.div(end, 2 * m, rounding_mode="floor"))


def _powerlaw(g, n, dmin):
    """Configuration model with P(k) ~ k^-2.3 on dmin..min(20000, n / 8), half-edges matched at random."""
    dmax = min(20000, max(dmin + 1, n // 8))
    w = torch.arange(dmin, dmax + 1, dtype=torch.float64, device="cuda") ** -2.3
    cdf = torch.cumsum(w, 0) / w.sum()
    d = dmin + torch.searchsorted(cdf, torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    d = d.clamp(max=dmax)
    stubs = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    stubs = stubs[torch.randperm(stubs.numel(), generator=g, device="cuda")]
    h = stubs.numel() // 2
    return _csr(n, stubs[:h], stubs[h:2 * h])


def _ws_batch(g, graphs, kmax):
    """Watts-Strogatz graphs, n uniform in [200, 20000], k even in [4, kmax], rewiring 0.1; one CSR and the offsets.
    The graphs' sizes depend on their number only (the outputs' length is the same for every seed)."""
    sizes = _rng(graphs)
    ns = torch.randint(200, 20001, (graphs,), generator=sizes, device="cuda")
    half = torch.randint(2, kmax // 2 + 1, (graphs,), generator=sizes, device="cuda")
    off = torch.zeros(graphs + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(ns, 0)
    per = ns * half
    gid = torch.repeat_interleave(torch.arange(graphs, device="cuda"), per)
    i = torch.arange(gid.numel(), device="cuda") - (torch.cumsum(per, 0) - per)[gid]
    local, step = torch.div(i, half[gid], rounding_mode="floor"), i % half[gid] + 1
    to = (local + step) % ns[gid]
    moved = torch.rand(i.numel(), generator=g, device="cuda") < 0.1
    other = (torch.rand(i.numel(), generator=g, device="cuda", dtype=torch.float64) * ns[gid]).to(torch.int64)
    to = torch.where(moved, other, to)
    base = off[gid]
    n = int(off[-1])
    rp, ci = _csr(n, base + local, base + to)
    return rp, ci, off.cpu().numpy()


def _graph(case, seed):
    g = _rng(seed)
    make = {"er": _erdos_renyi, "rmat": _rmat, "ba": _barabasi_albert, "plcm": _powerlaw, "ws": _ws_batch}
    return make[case["graph"]](g, case["n"], case["degree"])


def _watch_list(case, seed):
    return torch.randint(case["n"], (case["k"],), generator=_rng(seed + 1), device="cuda").to(torch.int32)


# ----------------------------------------------------------------- network

def _features(case, seed):
    """Rows like ef_features': sixteen logarithms of correlated counts, and EF-like targets."""
    g = _rng(seed)
    base = torch.randn(case["n"], 1, generator=g, device="cuda")
    x = 4.0 + 1.2 * base + 0.5 * torch.randn(case["n"], 16, generator=g, device="cuda")
    y = 5.0 + 0.8 * base[:, 0] + 0.1 * torch.randn(case["n"], generator=g, device="cuda")
    return x.contiguous(), y.contiguous()


def _weights(seed):
    """Flattened parameters of the 16-64-64-1 network and the features' mean and deviation."""
    g = torch.Generator().manual_seed(0xA11CE + seed)
    parts = [torch.randn(16 * 64, generator=g) / 4, 0.1 * torch.randn(64, generator=g),
             torch.randn(64 * 64, generator=g) / 8, 0.1 * torch.randn(64, generator=g),
             torch.randn(64, generator=g) / 8, 5.0 + 0.1 * torch.randn(1, generator=g),
             torch.full((16,), 4.0), torch.full((16,), 1.3)]
    return torch.cat(parts)


def _rank_weights():
    """A network that scores a node by its omega, S and degree features (a trained one does much the same)."""
    w1, w2, w3 = torch.zeros(16, 64), torch.zeros(64, 64), torch.zeros(64)
    for j, f in enumerate((3, 13, 1, 0)):
        w1[f, j] = 1.0
        w2[j, :] = 0.25
    w3[:] = 1.0 / 64
    mean = torch.tensor([2.2, 4.5, 7.0, 8.0, 2.5, 2.2, 1.5, 4.0, 4.6, 7.5, 3.0, 0.3, 0.01, 7.5, 2.5, 3.0]) - 2.0
    parts = [w1.flatten(), torch.zeros(64), w2.flatten(), torch.zeros(64), w3, torch.zeros(1), mean,
             torch.full((16,), 1.0)]
    return torch.cat(parts)


# --------------------------------------------------------------------- calls

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "ctx": ef.Context(0)}
    if kind in ("forward", "grad"):
        s["x"], s["y"] = _features(case, seed)
        s["model"] = ef.Model(s["ctx"].handle)
        s["model"].set(_weights(seed).numpy())
        s["out"] = torch.empty(case["n"], device="cuda")
        return s
    if kind == "batch":
        s["rp"], s["ci"], s["off"] = _graph(case, seed)
        s["ef"] = torch.empty(s["rp"].numel() - 1, dtype=torch.float64, device="cuda")
        return s
    s["rp"], s["ci"] = _graph(case, seed)
    if kind == "compute" and case["replay"] and case["n"] > 200_000:
        # a program that repeats a large call keeps its output buffers
        n = case["n"]
        s["out"] = {k: torch.empty(n, dtype=OUT_TYPES[k], device="cuda") for k in case["outputs"].split(",")}
    elif kind == "host":
        s["rp"], s["ci"] = s["rp"].cpu().pin_memory(), s["ci"].cpu().pin_memory()
        s["ef"] = torch.empty(case["n"], dtype=torch.float64).pin_memory()
    elif kind == "nodes":
        s["nodes"] = _watch_list(case, seed)
        s["out"] = {k: torch.empty(case["k"], dtype=OUT_TYPES[k], device="cuda") for k in ("ef", "s", "triangles")}
    elif kind == "sir":
        s["index"] = _watch_list(case, seed)
        s["beta"] = 1.3 / (3 * max(1.0, s["ci"].numel() / case["n"]))
        s["seed"] = seed
    elif kind == "rank":
        s["model"] = ef.Model(s["ctx"].handle)
        s["model"].set(_rank_weights().numpy())
        top = math.ceil(0.01 * case["n"]) + 1
        s["idx"] = torch.zeros(top, dtype=torch.int32, device="cuda")
        s["ef"] = torch.zeros(top, dtype=torch.float64, device="cuda")
        s["score"] = torch.empty(case["n"], device="cuda")
    return s


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "forward":
        state["model"].forward(state["x"], state["out"])
        return state["out"]
    if kind == "grad":
        loss, grad = state["model"].grad(state["x"], state["y"])
        return {"loss": loss, "grad": grad}
    rp, ci = state["rp"], state["ci"]
    if kind == "compute":
        replay = case["replay"]
        if "out" in state:
            ef.ef_compute_ex(ctx.handle, rp, ci, precision=case["precision"], device_check=replay, graph=replay,
                             **state["out"])
            return state["out"]
        return ctx.compute(rp, ci, precision=case["precision"], outputs=tuple(case["outputs"].split(",")),
                           device_check=replay, graph=replay)
    if kind == "host":
        ef.ef_compute_ex(ctx.handle, rp, ci, precision=case["precision"], ef=state["ef"], host_io=True)
        return state["ef"]
    if kind == "batch":
        ef.ef_compute_batched(ctx.handle, rp, ci, state["off"], precision=case["precision"], ef=state["ef"],
                              device_check=True, graph=True)
        return state["ef"]
    if kind == "nodes":
        ef.ef_compute_nodes(ctx.handle, rp, ci, state["nodes"], precision=case["precision"], **state["out"])
        return state["out"]
    if kind == "sir":
        return ctx.sir(rp, ci, state["index"], beta=state["beta"], gamma=1 / 3, seed=state["seed"],
                       outputs=("final_size", "length", "peak_infected", "peak_step", "spread", "spread_sims"))
    st = state["model"].rank(rp, ci, state["idx"], state["ef"], precision=case["precision"],
                             out_score=state["score"])
    return {"idx": state["idx"], "ef": state["ef"], "score": state["score"],
            "n_candidates": st["n_candidates"], "n_audit": st["n_audit"]}


# ---------------------------------------------------------------------- work

def _sizes(case):
    """Expected nodes and entries of a case's graph."""
    n, d = case["n"], case["degree"]
    if case["graph"] == "ws":
        return 10_100 * n, 10_100 * n * 8
    if case["graph"] == "plcm":
        dmax = min(20000, max(d + 1, n // 8))
        k = torch.arange(d, dmax + 1, dtype=torch.float64)
        return n, int(n * float((k ** -1.3).sum() / (k ** -2.3).sum()))
    return n, n * d


def work(case):
    """The graph (or rows) read once, the outputs written once; two operations per entry, or the network's products."""
    kind, n = case["kind"], case["n"]
    if kind in ("forward", "grad"):
        flops = 2 * n * (16 * 64 + 64 * 64 + 64)
        if kind == "forward":
            return {"bytes": 68 * n + 21_380, "flops": flops}
        return {"bytes": 68 * n + 2 * 21_380, "flops": 3 * flops}
    n, m = _sizes(case)
    graph = 4 * (n + 1) + 4 * m
    if kind == "compute":
        out = n * sum(OUT_TYPES[k].itemsize for k in case["outputs"].split(","))
    elif kind in ("host", "batch"):
        out = 8 * n
    elif kind == "nodes":
        out = 28 * case["k"]
    elif kind == "sir":
        out = 16 * case["k"] + 40 * n
    else:
        out = 4 * n + 12 * math.ceil(0.01 * n)
    return {"bytes": graph + out, "flops": 2 * m}


# --------------------------------------------------------------------- exact

CHUNK = 1 << 26


def _chunks(sizes):
    """Ranges [a, b) of consecutive items whose sizes add up to about CHUNK at most."""
    total = torch.cumsum(sizes, 0)
    a, done = 0, 0
    while a < sizes.numel():
        b = max(a + 1, int(torch.searchsorted(total, done + CHUNK, right=True)))
        yield a, b
        a, done = b, int(total[b - 1])


def _exact_ef(rp, ci):
    """EF, N, S, T, triangles and flags of every node in 64 bits: clusters by classes of equal neighbour degree,
    triangles by testing the pairs of each node's higher-ranked neighbours."""
    n, dev = rp.numel() - 1, rp.device
    rp, ci = rp.long(), ci.long()
    D = rp[1:] - rp[:-1]
    row = torch.repeat_interleave(torch.arange(n, device=dev), D)
    Dx = D[ci]
    top = 3 * int(D.max()) + 1
    d = torch.arange(top, dtype=torch.float64, device=dev)
    f = torch.where(d > 1, d * torch.log(d.clamp(min=1)), torch.zeros_like(d))
    # classes (node, neighbour degree) with their counts
    width = int(D.max()) + 1
    key, cls, count = torch.unique(row * width + Dx, return_inverse=True, return_counts=True)
    cu = torch.div(key, width, rounding_mode="floor")
    cb = key - cu * width
    K = torch.bincount(cu, minlength=n)
    first = torch.cumsum(K, 0) - K
    Q = torch.empty(key.numel(), dtype=torch.float64, device=dev)
    per = K[cu]
    for a, b in _chunks(per):
        k = per[a:b]
        i = torch.repeat_interleave(torch.arange(a, b, device=dev), k)
        j = torch.arange(i.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k) + first[cu[i]]
        at = (D[cu[i]] - 4 + cb[i] + cb[j]).clamp(min=0)
        Q[a:b] = torch.segment_reduce(count[j] * f[at], "sum", lengths=k)
    R = Q[cls] - f[(D[row] - 4 + 2 * Dx).clamp(min=0)]
    sig1 = torch.zeros(n, dtype=torch.int64, device=dev).index_add_(0, row, Dx)
    RS = (D[row] - 1) * (D[row] - 4 + Dx) + sig1[row] - Dx
    T = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, row, R).index_add_(0, ci, R)
    S = torch.zeros(n, dtype=torch.int64, device=dev).index_add_(0, row, RS).index_add_(0, ci, RS)
    N = D * (D - 1) + sig1 - D
    del R, RS, Q, cls, key, cu, cb, count, per
    # triangles, each at its lowest-ranked node in (degree, id)
    out = (D[row] < Dx) | ((D[row] == Dx) & (row < ci))
    src, dst = row[out], ci[out]
    del row, Dx, out
    code = src * n + dst
    left = torch.bincount(src, minlength=n).cumsum(0)[src] - torch.arange(src.numel(), device=dev) - 1
    t = torch.zeros(n, dtype=torch.int64, device=dev)
    for a, b in _chunks(left):
        k = left[a:b]
        e = torch.repeat_interleave(torch.arange(a, b, device=dev), k)
        if e.numel() == 0:
            continue
        c = e + 1 + torch.arange(e.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
        x, y = dst[e], dst[c]
        low = (D[x] < D[y]) | ((D[x] == D[y]) & (x < y))
        want = torch.where(low, x * n + y, y * n + x)
        at = torch.searchsorted(code, want).clamp(max=code.numel() - 1)
        hit = torch.nonzero(code[at] == want).squeeze(1)
        x, y, u = x[hit], y[hit], src[e[hit]]
        total = D[x] + D[y] + D[u]
        g = 4 * (f[total - 6] - f[total - 4])
        for v in (x, y, u):
            T.index_add_(0, v, g)
            t += torch.bincount(v, minlength=n)
    S = S - 8 * t
    some = S > 0
    Sd = torch.where(some, S, torch.ones_like(S)).double()
    e = torch.where(some, torch.log(Sd) - T / Sd, torch.zeros_like(T))
    return {"ef": e, "n_clusters": N, "s": S, "t": T, "triangles": t, "flag": (~some).to(torch.uint8)}


def _exact_network(case, seed):
    x, y = _features(case, seed)
    w = _weights(seed).double().cuda()
    p = w[:5313].clone().requires_grad_(case["kind"] == "grad")
    w1, b1, w2 = p[:1024].view(16, 64), p[1024:1088], p[1088:5184].view(64, 64)
    b2, w3, b3 = p[5184:5248], p[5248:5312], p[5312]
    z = (x.double() - w[5313:5329]) / w[5329:5345]
    score = torch.relu(torch.relu(z @ w1 + b1) @ w2 + b2) @ w3 + b3
    if case["kind"] == "forward":
        return score
    loss = ((score - y.double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": p.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        return _exact_network(case, seed)
    if kind in ("sir", "rank"):
        return None
    got = _exact_ef(*_graph(case, seed)[:2])
    if kind == "compute":
        return {k: got[k] for k in case["outputs"].split(",")}
    if kind == "nodes":
        at = _watch_list(case, seed).long()
        return {k: got[k][at] for k in ("ef", "s", "triangles")}
    return got["ef"]
