"""Performance cases: what a user of the library has it do, through the Python
binding and the C ABI, over the range of graphs, tree sizes, count widths and
options it is used with.

A case is a dict of plain values; see KINDS below for what one pass does.
Inputs are generated on the GPU from the seed alone, with the families the
benchmark uses (Erdos-Renyi, Chung-Lu power laws, R-MAT, road-like grids);
both the graph and the colouring change with the seed.
"""
import math

import numpy as np
import torch

import paper_2009_03052_gb300 as M

KINDS = ("count", "build", "rebuild", "batch", "sample", "ags", "packed")

# rooted treelet shapes on h nodes, h = 0..8 (0: none)
ROOTED = (0, 1, 1, 2, 4, 9, 20, 48, 115)


def listed():
    return [
        # the smallest whole job: load a tiny graph from host memory (checked),
        # colour, build, 10k samples, estimates -- launches, allocations and
        # synchronisations count, not bytes
        dict(name="count_er_1k_k4", kind="count", family="er", n=1000, m=4000, k=4, bits=64,
             samples=10_000, trusted=False),
        # the benchmark's job end to end: a social graph of 1M nodes from pinned
        # host memory, colour, build, 1M samples, estimates
        dict(name="count_chung_lu_1m_k5", kind="count", family="chung_lu", n=1_000_000, m=10_000_000,
             gamma=2.5, k=5, bits=64, samples=1_000_000, trusted=True),
        # the same job with round skipping: level k-1 never built, stars sampled
        # uncoloured (the memory saver for the largest k); a ragged node count
        dict(name="count_skip_chung_lu_100k_k6", kind="count", family="chung_lu", n=100_003, m=1_000_000,
             gamma=2.3, k=6, bits=128, samples=200_000, trusted=False, skip_round=True),
        # a road network (degrees of at most 8, no hubs), 64-bit counts
        dict(name="build_grid_1m_k6", kind="build", family="grid", side=997, k=6, bits=64),
        # many colourings of one graph: the build again in place per colouring
        # (the batch workload's 200k-node graph)
        dict(name="rebuild_chung_lu_200k_k6", kind="rebuild", family="chung_lu", n=200_000, m=2_000_000,
             gamma=2.3, k=6, bits=128),
        # a large heavy-tailed graph, fresh tables of 41 GB with 128-bit counts
        dict(name="build_rmat_22_k7", kind="build", family="rmat", scale=22, edge_factor=16, k=7, bits=128),
        # the largest k, fresh tables of 64 GB with 128-bit counts
        dict(name="build_chung_lu_2m_k8", kind="build", family="chung_lu", n=2_000_000, m=20_000_000,
             gamma=2.5, k=8, bits=128),
        # many uneven small graphs built in one pass over their disjoint union
        dict(name="batch_32_graphs_k6", kind="batch", graphs=32, n_lo=1000, n_hi=100_000, sizes=7, k=6,
             bits=128),
        # drawing classified samples from resident tables, a large request
        dict(name="sample_chung_lu_1m_k5", kind="sample", family="chung_lu", n=1_000_000, m=10_000_000,
             gamma=2.5, k=5, bits=64, h=5, samples=1_000_000),
        # a small serving request on the tables of the largest k: latency
        dict(name="sample_1k_chung_lu_300k_k8", kind="sample", family="chung_lu", n=300_000, m=3_000_000,
             gamma=2.5, k=8, bits=128, h=8, samples=1000),
        # adaptive graphlet sampling from resident tables
        dict(name="ags_rmat_19_k7", kind="ags", family="rmat", scale=19, edge_factor=16, k=7, bits=128, h=7,
             samples=2_000_000, cbar=1000),
        # a biased colouring with variable-length succinct tables (what the bias
        # is for), then samples from the packed rows
        dict(name="packed_chung_lu_200k_k6", kind="packed", family="chung_lu", n=200_000, m=2_000_000,
             gamma=2.3, k=6, bits=128, samples=200_000, bias=0.08, varlen=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "batch":
        return dict(kind="batch", graphs=rng.randint(2, 40), n_lo=_log_int(rng, 100, 2000),
                    n_hi=_log_int(rng, 5000, 100_000), sizes=rng.randint(0, 999), k=rng.randint(3, 6), bits=128)
    c = dict(kind=kind)
    k = rng.randint(4, 8)
    c["family"] = rng.choice(("er", "chung_lu", "rmat", "grid"))
    # 64-bit counts where they are wide enough for the family's degrees
    wide = 6 if c["family"] in ("er", "grid") else 5
    c["bits"] = rng.choice((64, 128)) if k <= wide else 128
    c["k"] = k
    # tables of at most 4 GB, at most 2M nodes
    top = min(2_000_000, int(4e9 / (c["bits"] // 8 * sum(_widths(k)))))
    if c["family"] == "rmat":
        c["scale"] = rng.randint(10, int(math.log2(top)))
        c["edge_factor"] = rng.randint(4, 16)
    elif c["family"] == "grid":
        c["side"] = _log_int(rng, 31, int(math.sqrt(top)))
    else:
        c["n"] = _log_int(rng, 1000, top)
        c["m"] = c["n"] * rng.randint(4, 20) // 2
        if c["family"] == "chung_lu":
            c["gamma"] = round(rng.uniform(2.2, 2.8), 2)
    if kind == "build":
        c["zero_root"] = rng.random() < 0.25
    if kind == "count":
        c["trusted"] = rng.random() < 0.5
        c["samples"] = _log_int(rng, 1000, 1_000_000)
        c["skip_round"] = rng.random() < 0.25
    if kind == "sample":
        c["h"] = rng.randint(max(3, k - 2), k)
        c["samples"] = _log_int(rng, 1000, 1_000_000)
    if kind == "ags":
        c["h"] = k
        c["samples"] = _log_int(rng, 100_000, 1_000_000)
        c["cbar"] = 1000
    if kind == "packed":
        c["samples"] = _log_int(rng, 1000, 200_000)
        c["varlen"] = rng.random() < 0.5
        c["bias"] = round(rng.choice((0.0, 0.5 / k)), 3)
    return c


# ---------------------------------------------------------------------------
# graphs, made on the GPU
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _csr(n, a, b):
    """Canonical CSR (symmetric, sorted, no loops or duplicates): int64
    row_ptr[n + 1], 32-bit col."""
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.cat([a * n + b, b * n + a])
    del a, b, keep
    key = torch.sort(key).values
    if key.numel():
        first = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
        first[1:] = key[1:] != key[:-1]
        key = key[first]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return row_ptr, (key % n).to(torch.int32)


def _chung_lu(n, m, gamma, g):
    """m endpoint pairs drawn in proportion to (i + i0)^(-1/(gamma-1)), the top
    expected degree 10k (n / 1M)^(2/3) (the benchmark's family), ids shuffled."""
    al = 1.0 / (gamma - 1.0)
    top = max(10_000.0 * (n / 1e6) ** (2.0 / 3.0), 20.0)
    lo, hi = 1e-9, float(n)
    for _ in range(100):
        mid = math.sqrt(lo * hi)
        mass = ((n + mid) ** (1 - al) - mid ** (1 - al)) / (1 - al) + 0.5 * mid ** -al
        lo, hi = (mid, hi) if 2.0 * m * mid ** -al / mass > top else (lo, mid)
    cdf = torch.cumsum((torch.arange(n, dtype=torch.float64, device="cuda") + hi) ** -al, 0)
    cdf /= cdf[-1].clone()
    ab = torch.searchsorted(cdf, torch.rand(2 * m, generator=g, dtype=torch.float64, device="cuda"))
    ab = torch.randperm(n, generator=g, device="cuda")[ab.clamp_(max=n - 1)]
    return ab[:m], ab[m:]


def _rmat(scale, edge_factor, g):
    n, m = 1 << scale, edge_factor << scale
    parts = []
    for s0 in range(0, m, 1 << 24):
        cnt = min(1 << 24, m - s0)
        u = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        v = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        for bit in range(scale):
            r = torch.rand(cnt, generator=g, device="cuda")
            down = r >= 0.76
            right = ((r >= 0.57) & ~down) | (r >= 0.95)
            u |= down.to(torch.int64) << bit
            v |= right.to(torch.int64) << bit
        parts.append((u, v))
    perm = torch.randperm(n, generator=g, device="cuda")
    return perm[torch.cat([p[0] for p in parts])], perm[torch.cat([p[1] for p in parts])]


def _grid(side, g):
    """side x side grid, 10% of its edges deleted, 2% of the diagonals added."""
    idx = torch.arange(side * side, device="cuda").reshape(side, side)
    ends = [(idx[:, :-1], idx[:, 1:], 0.9), (idx[:-1], idx[1:], 0.9), (idx[:-1, :-1], idx[1:, 1:], 0.02)]
    a, b = [], []
    for x, y, p in ends:
        keep = torch.rand(x.numel(), generator=g, device="cuda") < p
        a.append(x.reshape(-1)[keep])
        b.append(y.reshape(-1)[keep])
    return torch.cat(a), torch.cat(b)


def _graph(c, g):
    f = c["family"]
    if f == "rmat":
        return _csr(1 << c["scale"], *_rmat(c["scale"], c["edge_factor"], g))
    if f == "grid":
        return _csr(c["side"] ** 2, *_grid(c["side"], g))
    if f == "chung_lu":
        return _csr(c["n"], *_chung_lu(c["n"], c["m"], c["gamma"], g))
    ab = torch.randint(0, c["n"], (2, c["m"]), generator=g, device="cuda")
    return _csr(c["n"], ab[0], ab[1])


def _batch_sizes(c):
    """Node counts (log-uniform), average degrees and families of a batch."""
    rng = np.random.default_rng(c["sizes"])
    out = []
    for i in range(c["graphs"]):
        n = int(np.exp(rng.uniform(np.log(c["n_lo"]), np.log(c["n_hi"]))))
        m = int(n * rng.uniform(4, 20) / 2)
        out.append(dict(family="er", n=n, m=m) if i % 2 == 0 else dict(family="chung_lu", n=n, m=m, gamma=2.3))
    return out


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _read(T, h, n):
    """Level h of the count table as the C ABI copies it to device memory:
    64-bit words, two per count (low first) for 128-bit counts."""
    W, size = T.layout(h)
    out = torch.empty(n * W * (size // 8), dtype=torch.int64, device="cuda")
    M._check(M.load().mc_read_table(T.handle, h, 0, out.data_ptr(), out.numel() * 8, 1,
                                    torch.cuda.current_stream().cuda_stream))
    return out


def _words(x):
    return np.array([(x >> (32 * i)) & 0xffffffff for i in range(4)], dtype=np.int64)


def _bias(c):
    return int(c.get("bias", 0.0) * 2 ** 32)


def prepare(case, seed):
    c, g = case, _generator(seed)
    st = {"case": c, "seed": int(seed)}
    if c["kind"] == "batch":
        st["graphs"] = [M.Graph(*_graph(s, g)) for s in _batch_sizes(c)]
        st["colors"] = [M.color(G, c["k"], seed + i) for i, G in enumerate(st["graphs"])]
        return st
    row_ptr, col = _graph(c, g)
    if c["kind"] == "count":  # a program that has read its graph into page-locked memory
        st["row_ptr"], st["col"] = row_ptr.cpu().pin_memory(), col.cpu().pin_memory()
        M.sigma(c["k"])
        return st
    G = st["G"] = M.Graph(row_ptr, col)
    if c["kind"] in ("sample", "ags", "rebuild"):
        st["T"] = M.Tables(G, M.color(G, c["k"], seed), c["k"], c["bits"])
    if c["kind"] == "rebuild":  # the next colouring
        st["colors"] = M.color(G, c["k"], seed + 1)
    if c["kind"] == "sample":
        M.num_classes(c["h"])
        st["T"].total(c["h"])
    if c["kind"] in ("ags", "packed"):
        M.sigma(c["k"])
    torch.cuda.synchronize()
    return st


def run(state):
    c, seed = state["case"], state["seed"]
    kind, k = c["kind"], c["k"]
    if kind == "batch":
        T, offsets = M.Tables.batch(state["graphs"], state["colors"], k, c["bits"])
        return {"table": _read(T, k, int(offsets[-1])), "offsets": offsets}
    if kind == "count":
        G = M.Graph(state["row_ptr"], state["col"], trusted=c["trusted"])
        skip = c.get("skip_round", False)
        T = M.Tables(G, M.color(G, k, seed), k, c["bits"], skip_round=skip)
        est, hits, _ = T.estimate(k, seed=seed, samples=c["samples"], star_samples=c["samples"] if skip else 0)
        total = T.total(k)
        T.free()
        G.free()
        return {"est": est, "hits": hits.astype(np.int64), "rooted": _words(total[0]), "total": _words(total[1])}
    G = state["G"]
    if kind == "build":
        T = M.Tables(G, M.color(G, k, seed), k, c["bits"], zero_root=c.get("zero_root", False))
        return {"table": _read(T, k, G.n)}
    if kind == "rebuild":
        T = state["T"]
        T.rebuild(state["colors"])
        T.status()
        return {"table": _read(T, k, G.n)}
    if kind == "sample":
        nodes, roots, shapes, classes = state["T"].sample(c["h"], seed, 0, c["samples"])
        return {"nodes": nodes, "roots": roots, "shapes": shapes, "classes": classes}
    if kind == "ags":
        est, hits, stats = state["T"].estimate(c["h"], seed=seed, samples=c["samples"], mode=M.MC_EST_AGS,
                                               cbar=c["cbar"])
        return {"est": est, "hits": hits.astype(np.int64),
                "stats": [stats[s] for s in ("samples", "switches", "covered")]}
    T = M.Tables(G, M.color(G, k, seed, bias_q32=_bias(c)), k, c["bits"], succinct=True, varlen=c["varlen"])
    est, hits, _ = T.estimate(k, seed=seed, samples=c["samples"], colour_bias_q32=_bias(c))
    return {"est": est, "hits": hits.astype(np.int64), "table": _read(T, k, G.n)}


def exact(case, seed):
    # Tables, samples and hits are whole numbers.  The estimates are one
    # correctly rounded formula of the hits of this library's own random
    # samples, which no computation without them gives.
    return None


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _widths(k, skip=False):
    """Entries per node of every kept level: counts c_2..c_k, sums S_1..S_(k-1)."""
    hs = [h for h in range(1, k + 1) if not (skip and h == k - 1)]
    return [ROOTED[h] * math.comb(k - 1, h - 1) for h in hs if h > 1] + \
           [ROOTED[h] * math.comb(k - 1, h) for h in hs if h < k]


def _size(c):
    """Nodes and (about) adjacency entries."""
    if c["kind"] == "batch":
        n = c["graphs"] * (c["n_hi"] - c["n_lo"]) / math.log(c["n_hi"] / c["n_lo"])
        return n, 12 * n
    if c["family"] == "rmat":
        return 1 << c["scale"], 2 * c["edge_factor"] << c["scale"]
    if c["family"] == "grid":
        return c["side"] ** 2, 2 * c["side"] ** 2 * 1.82
    return c["n"], 2 * c["m"]


def work(case):
    """Bytes: the graph and the colours read once; every table entry written
    once and the level-k table copied out where a pass builds; per sample one
    32-byte sector for the root's prefix, and for each of the h - 1 steps one
    of a table row and one of an adjacency list, and its outputs.  The
    arithmetic is on integers: no floating-point operations."""
    c, k = case, case["k"]
    n, nnz = _size(c)
    graph, B = 8 * (n + 1) + 4 * nnz + n, c["bits"] // 8
    b = 0
    if c["kind"] not in ("sample", "ags"):
        b += graph + n * B * sum(_widths(k, c.get("skip_round", False)))
    if c["kind"] in ("build", "rebuild", "batch", "packed"):
        b += 2 * n * B * ROOTED[k]
    if "samples" in c:
        h = c.get("h", k)
        b += c["samples"] * (32 * (1 + 2 * (h - 1)) + (4 * h + 12 if c["kind"] == "sample" else 0))
    return {"bytes": b, "flops": 0}
