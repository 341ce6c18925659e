"""The work a user of this library has it do, as measurable cases.

A case names one public call and the graph it runs on:

  cluster    Graph.cluster on a resident graph (one clustering per pass)
  objective  Graph.disagreements of a given labelling on a resident graph
  oneshot    a host CSR clustered once: Graph(off, col), cluster, close
  batch      batch_jobs: many graphs, several orders each
  serve      a burst of requests through Server (submit all, wait for all)

Graphs are synthetic, made on the GPU from the seed: Erdos-Renyi, planted
partition, R-MAT and Chung-Lu, the four families of this repository's
benchmark and tests, in CSR form (off int64[n+1], col int32[nnz], symmetric,
rows sorted, no loops).
"""
import math

import numpy as np
import torch

import paper_1507_05086_gb300 as cc

MASK = (1 << 64) - 1


# ---- the cases -----------------------------------------------------------------

def listed():
    return [
        # the smallest graph of the benchmark, called as the README shows (host
        # labels): latency per round and per call
        {"name": "er10k_cw", "call": "cluster", "graph": "er", "n": 10_000, "degree": 20.0, "algo": "cw",
         "eps": 0.5, "labels": "host"},
        # a community graph (the benchmark's planted partition), small eps: many
        # short rounds
        {"name": "planted1m_cw_eps01", "call": "cluster", "graph": "planted", "n": 1_000_000, "algo": "cw",
         "eps": 0.1, "labels": "device"},
        # the same family, odd size, large eps: few wide rounds, many blocked
        # actives for C4's concurrency control
        {"name": "planted700k_c4_eps09", "call": "cluster", "graph": "planted", "n": 700_001, "algo": "c4",
         "eps": 0.9, "labels": "device"},
        # the practical schedule of the paper's Sec. 5: many rounds, binomial batches
        {"name": "rmat18_c4_est", "call": "cluster", "graph": "rmat", "scale": 18, "edge_factor": 16,
         "algo": "c4-est", "eps": 0.9, "labels": "device"},
        # C4 without rounds on a power-law graph
        {"name": "rmat22_c4_async", "call": "cluster", "graph": "rmat", "scale": 22, "edge_factor": 16,
         "algo": "c4-async", "eps": 0.5, "labels": "device"},
        # the benchmark's middle R-MAT size, serializable clustering
        {"name": "rmat24_c4", "call": "cluster", "graph": "rmat", "scale": 24, "edge_factor": 16, "algo": "c4",
         "eps": 0.5, "labels": "device"},
        # the headline: a billion-edge graph resident on the GPU
        {"name": "rmat26_cw", "call": "cluster", "graph": "rmat", "scale": 26, "edge_factor": 16, "algo": "cw",
         "eps": 0.5, "labels": "device"},
        # scoring a known labelling (the planted one) against the graph
        {"name": "objective_planted2m", "call": "objective", "graph": "planted", "n": 2_000_003},
        # a graph that is clustered once, from host memory to host labels
        {"name": "oneshot_rmat20_cw", "call": "oneshot", "graph": "rmat", "scale": 20, "edge_factor": 16,
         "algo": "cw", "eps": 0.5},
        # best-of-8 over many power-law graphs of uneven size
        {"name": "batch256_cw", "call": "batch", "graph": "chunglu", "count": 256, "n_lo": 1_000, "n_hi": 1_000_000,
         "orders": 8, "algo": "cw", "eps": 0.5},
        # the same with C4 and few small graphs: a batch that leaves most of the GPU idle
        {"name": "batch48_small_c4", "call": "batch", "graph": "chunglu", "count": 48, "n_lo": 1_000,
         "n_hi": 60_000, "orders": 3, "algo": "c4", "eps": 0.5},
        # a burst of requests of both algorithms over resident graphs
        {"name": "serve192", "call": "serve", "graph": "chunglu", "count": 64, "n_lo": 1_000, "n_hi": 400_000,
         "requests": 192, "eps": 0.5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["cluster"] * 5 + ["objective", "oneshot", "batch", "serve"])
    eps = rng.choice([0.1, 0.25, 0.5, 0.5, 0.9])
    if call in ("batch", "serve"):
        lo = rng.choice([300, 1_000, 5_000])
        c = {"call": call, "graph": "chunglu", "count": int(_log(rng, 16, 200)), "n_lo": lo,
             "n_hi": int(_log(rng, 20_000, 900_000)), "eps": max(eps, 0.25)}
        if call == "batch":
            c["orders"] = rng.randint(1, 8)
            c["algo"] = rng.choice(["cw", "c4"])
        else:
            c["requests"] = int(_log(rng, 24, 220))
        return c
    family = rng.choice(["er", "planted", "rmat", "rmat", "chunglu1"])
    c = {"call": call, "graph": family}
    if family == "er":
        c["n"] = int(_log(rng, 2_000, 800_000)) | 1
        c["degree"] = round(rng.uniform(6.0, 48.0), 2)
    elif family == "planted":
        c["n"] = int(_log(rng, 20_000, 2_000_000)) | 1
    elif family == "chunglu1":
        c["n"] = int(_log(rng, 5_000, 3_000_000)) | 1
        c["degree"] = round(rng.uniform(8.0, 64.0), 2)
    else:
        c["scale"] = rng.randint(14, 24)
        c["edge_factor"] = rng.randint(8, 20)
    if call == "objective":
        return c
    c["algo"] = rng.choice(["cw", "cw", "c4", "c4", "c4-async"])
    c["eps"] = eps
    if call == "cluster":
        small = c.get("n", 1 << c.get("scale", 0)) <= 400_000
        if small and rng.random() < 0.15:
            c["algo"] = rng.choice(["cw-est", "c4-est"])
            c["eps"] = 0.9
        c["labels"] = rng.choice(["device", "device", "host"])
    return c


# ---- graphs ----------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & ((1 << 62) - 1))
    return g


def _rand(shape, gen):
    return torch.rand(shape, device="cuda", generator=gen)


def _randint(n, shape, gen):
    return torch.randint(0, n, shape, device="cuda", generator=gen)


def _csr_of_keys(n, pieces):
    """CSR from pieces of keys row << 32 | column, the pieces in row order."""
    cols, counts = [], torch.zeros(n, dtype=torch.int64, device="cuda")
    for p in range(len(pieces)):
        k = torch.unique(pieces[p], sorted=True)
        pieces[p] = None
        cols.append((k & 0xFFFFFFFF).to(torch.int32))
        k >>= 32
        r, c = torch.unique_consecutive(k, return_counts=True)
        counts[r] = c
        del k, r, c
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=off[1:])
    return off, cols[0] if len(cols) == 1 else torch.cat(cols)


def _csr(n, u, v):
    keep = u != v
    u, v = u[keep], v[keep]
    return _csr_of_keys(n, [torch.cat([(u << 32) | v, (v << 32) | u])])


def _er(n, degree, seed):
    gen = _gen(seed)
    m = max(1, int(round(n * degree / 2)))
    return _csr(n, _randint(n, (m,), gen), _randint(n, (m,), gen))


def _planted(n, seed):
    """Clusters of Zipf(1.5) sizes (one per 500 vertices, at least 5), about
    27 neighbours inside the cluster (at most 0.27 of it), 4 n noise pairs.
    Also returns the planted labelling."""
    gen = _gen(seed)
    q = max(1, n // 500)
    w = torch.arange(1, q + 1, dtype=torch.float64, device="cuda").pow(-1.5)
    size = 5 + torch.floor((n - 5 * q) * w / w.sum()).to(torch.int64)
    size[0] += n - int(size.sum())
    start = torch.cumsum(size, 0) - size
    perm = torch.randperm(n, device="cuda", generator=gen)
    s = size.to(torch.float64)
    p = torch.clamp(30.0 / torch.clamp(s - 1, min=1.0), max=0.3) * 0.9
    m = torch.round(p * s * (s - 1) / 2).to(torch.int64)
    c = torch.repeat_interleave(torch.arange(q, device="cuda"), m)
    ends = []
    for _ in range(2):
        x = (_rand((c.numel(),), gen).to(torch.float64) * s[c]).to(torch.int64)
        ends.append(perm[start[c] + torch.minimum(x, size[c] - 1)])
    noise = [_randint(n, (4 * n,), gen) for _ in range(2)]
    off, col = _csr(n, torch.cat([ends[0], noise[0]]), torch.cat([ends[1], noise[1]]))
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    lab[perm] = perm[torch.repeat_interleave(start, size)].to(torch.int32)     # a member's id names the cluster
    return off, col, lab


def _rmat(scale, edge_factor, seed):
    """R-MAT (0.57, 0.19, 0.19, 0.05); duplicates and loops removed."""
    gen = _gen(seed)
    n, total = 1 << scale, edge_factor << scale
    top = min(3, scale)
    parts = 1 if total <= (1 << 28) else 1 << top
    pieces = [[] for _ in range(parts)]
    step = 1 << 26
    for e0 in range(0, total, step):
        m = min(step, total - e0)
        u = torch.zeros(m, dtype=torch.int64, device="cuda")
        v = torch.zeros(m, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = _rand((m,), gen)
            row = r >= 0.76
            u.mul_(2).add_(row)
            v.mul_(2).add_(((r >= 0.57) & ~row) | (r >= 0.95))
        keep = u != v
        u, v = u[keep], v[keep]
        k = torch.cat([(u << 32) | v, (v << 32) | u])
        del u, v, keep
        if parts == 1:
            pieces[0].append(k)
        else:
            b = k >> (32 + scale - top)
            for p in range(parts):
                pieces[p].append(k[b == p])
            del b
        del k
    for p in range(parts):
        pieces[p] = torch.cat(pieces[p])
    off, col = _csr_of_keys(n, pieces)
    if total > (1 << 28):
        torch.cuda.empty_cache()
    return off, col


def _chunglu(n, degree, seed):
    """Power-law weights (exponent 2.1) capped at sqrt(n d)."""
    gen = _gen(seed)
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda").pow(-1.0 / 1.1)
    w = torch.clamp(w * (degree * n / w.sum()), max=math.sqrt(n * degree))
    cdf = torch.cumsum(w, 0)
    m = max(1, int(round(n * degree / 2)))
    ends = [torch.clamp(torch.searchsorted(cdf, torch.rand(m, dtype=torch.float64, device="cuda", generator=gen) *
                                           cdf[-1], right=True), max=n - 1) for _ in range(2)]
    return _csr(n, *ends)


def _graph(case, seed):
    kind = case["graph"]
    if kind == "er":
        return _er(case["n"], case["degree"], seed)
    if kind == "planted":
        return _planted(case["n"], seed)[:2]
    if kind == "rmat":
        return _rmat(case["scale"], case["edge_factor"], seed)
    return _chunglu(case["n"], case["degree"], seed)


def _labelling(case, seed):
    """A graph and the labelling it is scored under: the planted one, else
    every vertex with its smallest neighbour (itself when that is smaller)."""
    if case["graph"] == "planted":
        return _planted(case["n"], seed)
    off, col = _graph(case, seed)
    n = off.numel() - 1
    lab = torch.arange(n, dtype=torch.int32, device="cuda")
    row = torch.nonzero(off[1:] > off[:-1]).flatten()
    lab[row] = torch.minimum(lab[row], col[off[row]])
    return off, col, lab


def _sizes(case):
    """The sizes of a batch: n log-uniform in [n_lo, n_hi], mean degree in
    [8, 64], spread evenly so that every seed has the same total work."""
    out = []
    for i in range(case["count"]):
        f = ((i * 0.6180339887498949) % 1.0, (i * 0.7548776662466927) % 1.0)
        out.append((int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** f[0])), 8.0 + 56.0 * f[1]))
    return out


# ---- prepare and run -----------------------------------------------------------------

def prepare(case, seed):
    call = case["call"]
    st = {"case": case, "seed": int(seed)}
    if call == "cluster":
        off, col = _graph(case, seed)
        st["graph"] = cc.Graph(off, col)
        st["labels"] = torch.empty(off.numel() - 1, dtype=torch.int32, device="cuda") \
            if case["labels"] == "device" else None
    elif call == "objective":
        off, col, lab = _labelling(case, seed)
        st["graph"] = cc.Graph(off, col)
        st["labels"] = lab
    elif call == "oneshot":
        off, col = _graph(case, seed)
        st["keep"] = (off.cpu().pin_memory(), col.cpu().pin_memory())
        st["off"], st["col"] = (t.numpy() for t in st["keep"])
    else:
        graphs = [cc.Graph(*_chunglu(n, d, seed + 1000 * i)) for i, (n, d) in enumerate(_sizes(case))]
        st["graphs"] = graphs
        st["seeds"] = np.arange(len(graphs), dtype=np.uint64) * np.uint64(64) + np.uint64(seed)
        if call == "serve":
            reqs = [(graphs[i % len(graphs)], ("cw", "c4")[(i // 3) % 2], seed + i) for i in range(case["requests"])]
            st["labels"] = torch.empty(sum(g.n for g, _, _ in reqs), dtype=torch.int32, device="cuda")
            at = np.concatenate([[0], np.cumsum([g.n for g, _, _ in reqs])])
            st["requests"] = [(g, a, s, st["labels"][at[i]:at[i + 1]]) for i, (g, a, s) in enumerate(reqs)]
            st["server"] = cc.Server()
    return st


def run(state):
    case, seed = state["case"], state["seed"]
    call = case["call"]
    if call == "cluster":
        labels, rounds, cost = state["graph"].cluster(case["algo"], case["eps"], seed, labels_out=state["labels"])
        return {"labels": labels, "rounds": rounds, "disagreements": cost}
    if call == "objective":
        return {"disagreements": state["graph"].disagreements(state["labels"])}
    if call == "oneshot":
        with cc.Graph(state["off"], state["col"]) as g:
            labels, rounds, cost = g.cluster(case["algo"], case["eps"], seed)
        return {"labels": labels, "rounds": rounds, "disagreements": cost}
    if call == "batch":
        cost, rounds = cc.batch_jobs(state["graphs"], case["algo"], case["eps"], state["seeds"], case["orders"])
        return {"rounds": rounds, "disagreements": cost}
    server = state["server"]
    tickets = [server.submit(g, a, case["eps"], s, labels_out=lab) for g, a, s, lab in state["requests"]]
    done = [server.wait(t)[:2] for t in tickets]
    return {"labels": state["labels"], "rounds": np.array([r for r, _ in done]),
            "disagreements": np.array([d for _, d in done])}


# ---- what a pass cannot do without ------------------------------------------------------

def _entries(case):
    """Vertices and CSR entries of the graph (expected; duplicates of R-MAT
    and Chung-Lu graphs left out approximately)."""
    kind = case["graph"]
    if kind == "rmat":
        n = 1 << case["scale"]
        return n, int(2 * case["edge_factor"] * n * (0.98 if case["scale"] >= 24 else 0.94))
    if kind == "planted":
        return case["n"], int(case["n"] * 34.4)
    return case["n"], int(case["n"] * case["degree"] * (0.9 if kind == "chunglu1" else 1.0))


def work(case):
    """Bytes: the CSR read once per clustering (offsets, columns) and the labels
    written once; flops: one comparison per CSR entry (integer work)."""
    if case["call"] in ("batch", "serve"):
        sizes = _sizes(case)
        if case["call"] == "serve":
            jobs = [sizes[i % len(sizes)] for i in range(case["requests"])]
            b = sum(8 * (n + 1) + 4 * 0.9 * n * d + 4 * n for n, d in jobs)
            return {"bytes": int(b), "flops": int(sum(0.9 * n * d for n, d in jobs))}
        k = case["orders"]
        b = sum(8 * (n + 1) + 4 * 0.9 * n * d for n, d in sizes) + 12 * k * len(sizes)
        return {"bytes": int(b), "flops": int(k * sum(0.9 * n * d for n, d in sizes))}
    n, nnz = _entries(case)
    return {"bytes": 8 * (n + 1) + 4 * nnz + 4 * n, "flops": nnz}


# ---- the same in plain numpy and torch ----------------------------------------------------

def _cost(off, col, lab):
    """Positive edges between clusters plus negative pairs inside them."""
    n = off.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=off.device), off[1:] - off[:-1])
    inside = int((lab[rows] == lab[col.long()]).sum())
    s = torch.bincount(lab.long(), minlength=n)
    return col.numel() // 2 - inside + int((s * (s - 1) // 2).sum())


def _order(n, seed):
    z = (np.arange(n, dtype=np.uint64) ^ np.uint64(seed & MASK)) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return np.argsort(z ^ (z >> np.uint64(31)), kind="stable")


def _rounds(off, col, order, wild, eps):
    """The paper's Alg. 2 round by round: C4, or ClusterWild! when wild."""
    n = off.size - 1
    ppm = int(round(eps * 1e6))
    src = np.repeat(np.arange(n), np.diff(off))
    lab = np.full(n, -1, np.int64)
    rounds, left = 0, order
    while left.size:
        alive = lab < 0
        both = alive[src] & alive[col]
        delta = int(np.bincount(src[both], minlength=n).max()) if both.any() else 0
        k = left.size if delta == 0 else min(left.size, -(-ppm * left.size // (1_000_000 * delta)))
        active = np.zeros(n, bool)
        active[left[:k]] = True
        for v in left[:k]:
            if lab[v] >= 0:
                continue
            lab[v] = v
            nb = col[off[v]:off[v + 1]]
            nb = nb[lab[nb] < 0]
            lab[nb[~active[nb]] if wild else nb] = v
        left = left[lab[left] < 0]
        rounds += 1
    return lab, rounds


def exact(case, seed):
    if case["call"] == "objective":
        off, col, lab = _labelling(case, seed)
        return {"disagreements": _cost(off, col, lab)}
    if case["call"] != "cluster" or case["algo"].endswith("-est"):
        return None
    n, nnz = _entries(case)
    if n > 30_000 or nnz > 1_000_000:
        return None
    off, col = _graph(case, seed)
    wild = case["algo"] == "cw"
    lab, rounds = _rounds(off.cpu().numpy(), col.cpu().numpy(), _order(n, int(seed)), wild, case["eps"])
    lab = torch.from_numpy(lab.astype(np.int32))
    return {"labels": lab, "rounds": 0 if case["algo"] == "c4-async" else rounds,
            "disagreements": _cost(off.cpu(), col.cpu(), lab)}
