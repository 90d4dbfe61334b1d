"""The work that users of the library have it do, as measurable cases.

A case names a graph family with its size, an entry point and its options.
prepare() draws the graph and the query vertices on the GPU from a seed and
creates the graph handle that a user's program keeps between calls; run() is
one call of the public entry point; exact() restates the call in 64 bits with
dense columns and plain torch operations.

Graphs: R-MAT with quadrant probabilities 0.57 / 0.19 / 0.19 / 0.05 (directed
power-law graphs with a giant strongly connected core and many small reach
sets), optionally with 30 % of the arcs also reversed (social links), and
directed Erdos-Renyi graphs. Weights are uniform integers.
"""
import gc
import math

import numpy as np
import torch

import paper_1708_08739_gb300 as bcd

DELTA = 0.1  # confidence of the sampled queries
QSEED = 7    # seed of their draws
KINDS = {"exact": bcd.BC_QUERY_EXACT, "approx": bcd.BC_QUERY_APPROX, "approx_T": bcd.BC_QUERY_APPROX_T,
         "hybrid": bcd.BC_QUERY_HYBRID}


def _case(op, graph, n, deg, recip=0.0, wmax=0, uniform=0, hubs=0, kind="exact", eps=0.0, T=0, name=None):
    c = {"op": op, "graph": graph, "n": n, "deg": deg, "recip": recip, "wmax": wmax, "uniform": uniform,
         "hubs": hubs, "kind": kind, "eps": eps, "T": T}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one vertex of a toy graph: launches and synchronisations
        _case("single", "er", 300, 5, kind="exact", name="single_exact_er300"),
        # the Erdos-Renyi configuration: 16 exact queries on 2,000 vertices
        _case("batch", "er", 2000, 8, uniform=16, kind="exact", name="batch16_exact_er2000"),
        # the reach set of one vertex of a large graph, read back by the host
        _case("rv", "rmat", 1 << 20, 16, name="rv_rmat20"),
        # the same inside a program that may not allocate, at the largest size it takes
        _case("rv_noalloc", "rmat", 1 << 22, 8, recip=0.3, name="rv_noalloc_rmat22"),
        # one vertex at a time with a fixed number of samples (1,000)
        _case("single", "rmat", 1 << 20, 16, kind="approx_T", T=1000, name="single_T1000_rmat20"),
        # exact scores of 32 uniform and 32 hub vertices, every source of a middle-sized graph
        _case("batch", "rmat", 1 << 16, 8, uniform=32, hubs=32, kind="exact", name="batch64_exact_rmat16"),
        # sampled scores of 32 uniform and 32 hub vertices of a large graph
        _case("batch", "rmat", 1 << 20, 16, uniform=32, hubs=32, kind="approx", eps=0.02, name="batch64_eps02_rmat20"),
        # the benchmark's batch (64 uniform vertices, reciprocal R-MAT 22) at the serving accuracy
        _case("batch", "rmat", 1 << 22, 8, recip=0.3, uniform=64, kind="approx", eps=0.02, name="batch64_eps02_rmat22"),
        # weights 1..255: 32 uniform vertices, sampled
        _case("batch", "rmat", 1 << 20, 16, wmax=255, uniform=32, kind="approx", eps=0.05, name="batch32_eps05_w255_rmat20"),
        # weights 1..255 with hub vertices among the queries: exact where the reach set is small, 1,000 samples elsewhere
        _case("batch", "rmat", 1 << 16, 16, wmax=255, uniform=32, hubs=32, kind="hybrid", T=1000,
              name="batch64_hybrid_w255_rmat16"),
        # continuous batching: 32 requests, half exact on small reach sets, half sampled
        _case("serve", "rmat", 1 << 22, 8, recip=0.3, uniform=32, kind="approx", eps=0.02, name="serve32_rmat22"),
        # one question about a graph that is still on the host: handle, answer, release
        _case("cold", "rmat", 1 << 18, 16, uniform=16, kind="hybrid", T=1000, name="cold16_hybrid_rmat18"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["single", "batch", "batch", "batch", "weighted", "weighted", "rv", "rv_noalloc", "serve", "cold"])
    graph = rng.choice(["er", "rmat", "rmat", "rmat"])
    recip = rng.choice([0.0, 0.3]) if graph == "rmat" else 0.0
    deg = rng.randint(4, 16)
    if op in ("rv", "rv_noalloc"):
        return _case(op, graph, _log(rng, 1000, 1 << 22 if op == "rv_noalloc" else 1 << 21), deg, recip)
    uniform, hubs = rng.randint(1, 40), rng.choice([0, 0, rng.randint(1, 24)])
    n = _log(rng, 300, 1 << 21)
    kind = rng.choice(["approx", "approx_T", "hybrid"] if n > 40000 else ["exact", "exact", "approx_T", "hybrid"])
    eps = rng.choice([0.02, 0.03, 0.05]) if kind == "approx" else 0.0
    T = _log(rng, 50, 2000) if kind in ("approx_T", "hybrid") else 0
    if op == "single":
        return _case(op, graph, n, deg, recip, kind="approx_T" if n > 40000 else kind, eps=eps, T=T or 1000)
    if op == "weighted":
        n = _log(rng, 300, 1 << 18)
        kind = "hybrid" if n > 10000 else "exact"
        return _case("batch", graph, n, deg, recip, wmax=rng.choice([15, 255, 1000]), uniform=uniform, hubs=hubs,
                     kind=kind, T=_log(rng, 50, 500))
    if op == "serve":
        return _case(op, "rmat", _log(rng, 20000, 1 << 21), deg, recip, uniform=rng.randint(4, 48), kind="approx",
                     eps=rng.choice([0.02, 0.05]))
    return _case(op, graph, n, deg, recip, uniform=uniform, hubs=hubs, kind=kind, eps=eps, T=T)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _graph(case, seed):
    """(offsets int64, cols int32, weights int32 or None) on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 17)
    n, m = case["n"], case["n"] * case["deg"]
    if case["graph"] == "er":
        t = torch.randint(0, n, (m,), device="cuda", generator=g)
        h = torch.randint(0, n, (m,), device="cuda", generator=g)
    else:
        # ids of the next power of two, those past n dropped
        t = torch.zeros(m, dtype=torch.int64, device="cuda")
        h = torch.zeros(m, dtype=torch.int64, device="cuda")
        for _ in range(max(1, (n - 1).bit_length())):
            u = torch.rand(m, device="cuda", generator=g)
            t = 2 * t + (u >= 0.76)
            h = 2 * h + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
            del u
        keep = (t < n) & (h < n)
        t, h = t[keep], h[keep]
    if case["recip"] > 0:
        back = torch.rand(t.shape[0], device="cuda", generator=g) < case["recip"]
        t, h = torch.cat([t, h[back]]), torch.cat([h, t[back]])
    key = torch.unique((t * n + h)[t != h])
    t, h = key // n, key % n
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(t, minlength=n), 0)
    w = None
    if case["wmax"]:
        w = torch.randint(1, case["wmax"] + 1, (h.shape[0],), device="cuda", generator=g).to(torch.int32)
    return off, h.to(torch.int32), w


def _reached(off, col, v):
    """Mask of the vertices that v reaches, v included (arc-parallel BFS)."""
    n = off.shape[0] - 1
    tail = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[v] = True
    count = 1
    while True:
        seen[col[seen[tail]].long()] = True
        now = int(seen.sum())
        if now == count:
            return seen
        count = now


def _vertices(case, seed, off, col):
    """The query vertices of a case, in query order."""
    rng = np.random.default_rng(seed + 5)
    n = case["n"]
    din = torch.bincount(col.long(), minlength=n)
    dout = off[1:] - off[:-1]
    prod = din * dout
    if case["op"] in ("single", "rv", "rv_noalloc"):
        # one well-connected vertex: among the first hundredth by in-degree x out-degree
        top = torch.argsort(prod, descending=True, stable=True)[: max(1, n // 100)]
        return [int(top[int(rng.integers(0, top.shape[0]))])]
    if case["op"] == "serve":
        # Zipf(1.1) popularity over the vertices with arcs both ways; every other request asks for a vertex that the
        # giant component does not reach (a small reach set, answered exactly)
        core = _reached(off, col, int(torch.argmax(prod)))
        big = torch.nonzero((prod > 0) & core).flatten().cpu().numpy()
        small = torch.nonzero((prod > 0) & ~core).flatten().cpu().numpy()
        small = small if small.shape[0] else big[-1:]
        out = []
        for i in range(case["uniform"]):
            ids = rng.permutation(small if i % 2 == 0 else big)
            p = np.arange(1, ids.shape[0] + 1, dtype=np.float64) ** -1.1
            out.append(int(ids[np.searchsorted(np.cumsum(p) / p.sum(), rng.random())]))
        return out
    hubs = torch.argsort(prod, descending=True, stable=True)[: case["hubs"]]
    return [int(x) for x in rng.integers(0, n, case["uniform"])] + [int(x) for x in hubs]


def _queries(case, vertices):
    out = []
    for i, r in enumerate(vertices):
        kind = case["kind"]
        if case["op"] == "serve" and i % 2 == 0:
            kind = "hybrid"  # exact up to 4,000 sources
        q = {"r": r, "kind": KINDS[kind]}
        if kind == "approx":
            q.update(eps=case["eps"], delta=DELTA, seed=QSEED)
        elif kind != "exact":
            q.update(T=4000 if case["op"] == "serve" else case["T"], seed=QSEED)
        out.append(q)
    return out


def prepare(case, seed):
    off, col, w = _graph(case, seed)
    queries = _queries(case, _vertices(case, seed, off, col))
    state = {"case": case, "queries": queries, "r": queries[0]["r"]}
    if case["op"] == "cold":
        # a program that has read its graph into pinned host memory
        host = [None if x is None else x.cpu().pin_memory() for x in (off, col, w)]
        state["host"] = host
        state["args"] = [None if x is None else x.numpy() for x in host]
        if w is not None:
            state["args"][2] = state["args"][2].view(np.uint32)
        return state
    g = bcd.bc_graph_create(case["n"], off, col, w)
    state["graph"] = g
    if case["op"] == "rv":
        state["rv"] = np.full(case["n"], -1, dtype=np.int32)
    elif case["op"] == "rv_noalloc":
        roff, rcol, _ = bcd.bc_graph_reverse(g)
        state["roff"], state["rcol"] = torch.from_numpy(roff).cuda(), torch.from_numpy(rcol.copy()).cuda()
        state["out"] = torch.full((case["n"],), -1, dtype=torch.int32, device="cuda")
    elif case["op"] == "serve":
        state["server"] = bcd.Server(g)
    del off, col, w
    gc.collect()
    torch.cuda.empty_cache()
    return state


# --------------------------------------------------------------------------
# one call
# --------------------------------------------------------------------------

def _answers(out):
    return {"bc": np.array([o["bc"] for o in out], dtype=np.float64),
            "rv_size": np.array([o["rv_size"] for o in out], dtype=np.int64),
            "samples": np.array([o["samples"] for o in out], dtype=np.int64),
            "flags": np.array([o["flags"] for o in out], dtype=np.int64),
            "status": np.array([o["status"] for o in out], dtype=np.int64)}


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "rv":
        # into the program's own array, -1 past the reach set
        rv = bcd.bc_rv_compute(state["graph"], state["r"])
        state["rv"][: rv.shape[0]] = rv
        return {"rv": state["rv"], "count": rv.shape[0]}
    if op == "rv_noalloc":
        k = bcd.bc_rv_compute_noalloc(state["roff"].data_ptr(), state["rcol"].data_ptr(), case["n"], state["r"],
                                      state["out"].data_ptr(), case["n"], torch.cuda.current_stream().cuda_stream)
        return {"rv": state["out"], "count": k}
    if op == "single":
        if case["kind"] == "exact":
            bc, info = bcd.bc_exact(state["graph"], state["r"])
        elif case["kind"] == "approx":
            bc, info = bcd.bc_approx(state["graph"], state["r"], case["eps"], DELTA, QSEED)
        elif case["kind"] == "approx_T":
            bc, info = bcd.bc_approx_T(state["graph"], state["r"], case["T"], QSEED)
        else:
            return _answers(bcd.bc_batch(state["graph"], state["queries"])[0])
        return _answers([{"bc": bc, "rv_size": info["rv_size"], "samples": info["samples"], "flags": info["flags"],
                          "status": 0}])
    if op == "serve":
        tickets = [state["server"].submit(q) for q in state["queries"]]
        out = []
        for t in tickets:
            got = None
            while got is None:
                got = state["server"].poll(t, timeout_us=10_000_000)
            out.append(got[0])
        return _answers(out)
    if op == "cold":
        g = bcd.bc_graph_create(case["n"], *state["args"])
        out, _ = bcd.bc_batch(g, state["queries"])
        g.close()
        return _answers(out)
    return _answers(bcd.bc_batch(state["graph"], state["queries"])[0])


# --------------------------------------------------------------------------
# what a call cannot do without
# --------------------------------------------------------------------------

def _samples(case):
    if case["op"] == "single" and case["kind"] == "exact" or case["kind"] == "exact":
        return case["n"]
    return math.ceil(math.log(2 / DELTA) / (2 * case["eps"] ** 2)) if case["kind"] == "approx" else case["T"]


def work(case):
    """Bytes: the graph once (both directions for the reach sets), the answers, and per single-source pass the level
    and path count of the vertices it reaches, written once and read once. Operations: per pass, one addition per arc
    forward and one for the dependencies."""
    n, m = case["n"], case["n"] * case["deg"] * (1 + case["recip"])
    part = 1.0 if case["graph"] == "er" else 0.5  # share of the vertices in the giant component
    graph = 8 * (n + 1) + 4 * m + (4 * m if case["wmax"] else 0)
    if case["op"] in ("rv", "rv_noalloc"):
        return {"bytes": graph + 4 * part * n, "flops": 0}
    passes = min(part * n, _samples(case))
    nq = max(1, case["uniform"] + case["hubs"])
    return {"bytes": 2 * graph + 40 * nq + passes * part * n * 2 * 12, "flops": 2 * passes * m}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _columns(case, off, col, w, sources, targets):
    """delta_s.(t) for every source s and target t [sources, targets], one dense column per source."""
    n, dev = case["n"], "cuda"
    m = int(col.shape[0])
    tail = torch.repeat_interleave(torch.arange(n, device=dev), off[1:] - off[:-1])
    head = col.long()
    S = sources.shape[0]
    at = torch.arange(S, device=dev)
    dist = torch.full((n, S), -1 if w is None else 1 << 40, dtype=torch.int64, device=dev)
    sigma = torch.zeros((n, S), dtype=torch.float64, device=dev)
    delta = torch.zeros((n, S), dtype=torch.float64, device=dev)
    dist[sources, at] = 0
    sigma[sources, at] = 1.0
    if w is None:
        ones = torch.ones(m, dtype=torch.float64, device=dev)
        out = torch.sparse_csr_tensor(off, head, ones, (n, n))
        order = torch.argsort(head, stable=True)
        roff = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        roff[1:] = torch.cumsum(torch.bincount(head, minlength=n), 0)
        inn = torch.sparse_csr_tensor(roff, tail[order], ones, (n, n))
        level = 0
        while True:
            reach = inn @ torch.where(dist == level, sigma, 0.0)
            new = (reach > 0) & (dist < 0)
            if not bool(new.any()):
                break
            level += 1
            dist[new] = level
            sigma[new] = reach[new]
        for k in range(level, 0, -1):
            c = torch.where(dist == k, (1.0 + delta) / sigma.clamp(min=1.0), 0.0)
            delta = torch.where(dist == k - 1, sigma * (out @ c), delta)
    else:
        wl = w.long()[:, None]
        while True:
            old = dist.clone()
            for a in range(0, m, 1 << 21):
                b = min(m, a + (1 << 21))
                dist.index_reduce_(0, head[a:b], old[tail[a:b]] + wl[a:b], "amin")
            if torch.equal(old, dist):
                break
        pairs = []
        for a in range(0, m, 1 << 21):
            b = min(m, a + (1 << 21))
            dt = dist[tail[a:b]]
            k, s = torch.nonzero((dt < 1 << 40) & (dt + wl[a:b] == dist[head[a:b]]), as_tuple=True)
            pairs.append((tail[a + k] * S + s, head[a + k] * S + s))
        pt, ph = torch.cat([p[0] for p in pairs]), torch.cat([p[1] for p in pairs])
        root, sg = sources * S + at, sigma.view(-1)
        while True:
            nxt = torch.zeros_like(sg).index_add_(0, ph, sg[pt])
            nxt[root] = 1.0
            if torch.equal(nxt, sg):
                break
            sg = nxt
        sigma, dl = sg.view(n, S), delta.view(-1)
        coef = sg[pt] / sg[ph]
        while True:
            nxt = torch.zeros_like(dl).index_add_(0, pt, coef * (1.0 + dl[ph]))
            # the order of the additions is not fixed: settled when nothing moves by more than rounding
            done = bool(((nxt - dl).abs() <= 1e-13 * nxt.abs()).all())
            dl = nxt
            if done:
                break
        delta = dl.view(n, S)
    got = delta[targets].T.clone()
    got[sources[:, None] == targets[None, :]] = 0.0
    return got


def exact(case, seed):
    off, col, w = _graph(case, seed)
    n = case["n"]
    queries = _queries(case, _vertices(case, seed, off, col))
    tail = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    order = torch.argsort(col, stable=True)
    roff = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    roff[1:] = torch.cumsum(torch.bincount(col.long(), minlength=n), 0)
    rcol = tail[order].to(torch.int32)

    def reach_set(r):
        seen = _reached(roff, rcol, r)
        seen[r] = False
        return torch.nonzero(seen).flatten()

    if case["op"] in ("rv", "rv_noalloc"):
        rv = reach_set(queries[0]["r"]).to(torch.int32)
        full = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        full[: rv.shape[0]] = rv
        return {"rv": full if case["op"] == "rv_noalloc" else full.cpu().numpy(), "count": int(rv.shape[0])}
    dout = off[1:] - off[:-1]
    kept, plans, need = {}, [], torch.zeros(n, dtype=torch.bool, device="cuda")
    for q in queries:
        r = q["r"]
        if int(dout[r]) == 0:
            plans.append((r, None, 0.0, 0, 0))
            continue
        if r not in kept:
            kept[r] = reach_set(r)
        rv = kept[r]
        k = int(rv.shape[0])
        T = math.ceil(math.log(2 / q["delta"]) / (2 * q["eps"] ** 2)) if q["kind"] == KINDS["approx"] else q.get("T", 0)
        if k == 0 or q["kind"] == KINDS["exact"] or (q["kind"] == KINDS["hybrid"] and k <= T):
            src, mult, scale, samples = rv, torch.ones(k, dtype=torch.float64, device="cuda"), 1.0, 0
        else:
            x = np.random.Philox(key=q["seed"], counter=2**256 - 1).random_raw(4 * T)[::4]
            lo, hi = x & np.uint64(0xFFFFFFFF), x >> np.uint64(32)
            idx = (hi * np.uint64(k) + ((lo * np.uint64(k)) >> np.uint64(32))) >> np.uint64(32)
            idx, mult = torch.unique(torch.from_numpy(idx.astype(np.int64)).cuda(), return_counts=True)
            src, mult, scale, samples = rv[idx], mult.double(), k / T, T
        need[src] = True
        plans.append((r, src, scale, k, samples))
        plans[-1] = plans[-1] + (mult,)
    union = torch.nonzero(need).flatten()
    if int(union.shape[0]) * int(col.shape[0]) > (1e11 if w is None else 4e9):
        return None
    targets = torch.tensor(sorted({q["r"] for q in queries}), device="cuda")
    S = max(1, min(256 if w is None else 64, int(3e9 / max(n, 1) / 8)))
    dep = torch.zeros((n, targets.shape[0]), dtype=torch.float64, device="cuda")
    for a in range(0, union.shape[0], S):
        dep[union[a:a + S]] = _columns(case, off, col, w, union[a:a + S], targets)
    bc, sizes, samples = [], [], []
    for p in plans:
        total = 0.0
        if p[1] is not None:
            j = int(torch.searchsorted(targets, p[0]))
            total = p[2] * float((dep[p[1], j] * p[5]).sum())
        bc.append(total)
        sizes.append(p[3])
        samples.append(p[4])
    return {"bc": np.array(bc), "rv_size": np.array(sizes, dtype=np.int64), "samples": np.array(samples, dtype=np.int64),
            "flags": None, "status": np.zeros(len(bc), dtype=np.int64)}
