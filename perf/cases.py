"""The calls this library is measured by.

A case is a seeded uncertain signed graph and one call of the Python package
on it: threshold counts, enumeration, top-k, expected counts with gradients,
sign worlds, a batch of small graphs, the end-to-end count from host arrays,
a build with the undirected rows and the edge index, and the two samplers.
Graphs are drawn with torch on the GPU in the structures and sizes of the
repository's configurations (Erdos-Renyi, Chung-Lu, R-MAT); their sign
probabilities follow the distributions the paper uses (Sec. 7).
"""
import math

import numpy as np
import torch

import paper_2602_14084_gb300 as ubt

ONE = 65536  # P+ = k / 65536


def listed():
    return [
        # the smallest call: three thresholds on G(2,000, 20,000), where launches and host work are everything
        dict(name="count_er2k", kind="count", graph="er", n=2000, draws=20000, dist="uniform", order="shuffled",
             n_tau=3, t_lo=0.6, t_hi=0.9, prune=True),
        # the ordinary query: a social network of a million vertices (power law), four thresholds, pruned
        dict(name="count_cl1m", kind="count", graph="cl", n=1000000, draws=10000000, gamma=2.1, dist="beta_half",
             order="sorted", n_tau=4, t_lo=0.55, t_hi=0.95, prune=True),
        # the largest query: R-MAT scale 22, a sweep of 32 thresholds in one traversal
        dict(name="count_rmat22", kind="count", graph="rmat", n=1 << 22, draws=16 << 22, dist="mixture", order="sorted",
             n_tau=32, t_lo=0.51, t_hi=0.99, prune=True),
        # listing the confident triangles of a mid-size graph, kept in (u, v, w) order
        dict(name="enumerate_rmat20", kind="enumerate", graph="rmat", n=1 << 20, draws=16 << 20, dist="mixture",
             order="sorted", t_lo=0.9, which=3, room=1 << 19),
        # one optimisation step on the probabilities: expected counts forward and backward
        dict(name="train_cl4m", kind="train", graph="cl", n=4000000, draws=40000000, edges=39000000, gamma=2.3,
             dist="real", order="sorted"),
        # Monte-Carlo: 4,096 bit-sliced sign worlds
        dict(name="worlds_rmat20", kind="worlds", graph="rmat", n=1 << 20, draws=16 << 20, dist="uniform",
             order="sorted", worlds=4096),
        # many small graphs of uneven size in one launch: counts, expected counts and 64 worlds of each
        dict(name="batch_1k", kind="batch", graphs=1000, s_lo=50, s_hi=5000, degree=100, dist="uniform",
             n_tau=3, t_lo=0.6, t_hi=0.9),
        # from host arrays to counts: copies, build, query (a graph that is asked once)
        dict(name="host_cl1m", kind="host", graph="cl", n=1000000, draws=10000000, gamma=2.1, dist="beta_half",
             order="sorted", n_tau=4, t_lo=0.55, t_hi=0.95, prune=True),
        # a new graph with everything Alg. 2 and the samplers need, and its first answer by Alg. 2
        dict(name="build_aeo_cl1m", kind="aeo", graph="cl", n=1000000, draws=10000000, gamma=2.1, dist="beta_half",
             order="sorted", n_tau=1, t_lo=0.9, t_hi=0.9),
        # edge sampling (Algs. 5-6): 10,000 samples, one threshold
        dict(name="sample_edges_cl1m", kind="sample", of="edges", graph="cl", n=1000000, draws=10000000, gamma=2.1,
             dist="beta_half", order="sorted", samples=10000, n_tau=1, t_lo=0.8, t_hi=0.8),
        # vertex sampling (Algs. 3-4): 10,000 samples, one threshold
        dict(name="sample_vertices_cl1m", kind="sample", of="vertices", graph="cl", n=1000000, draws=10000000,
             gamma=2.1, dist="beta_half", order="sorted", samples=10000, n_tau=1, t_lo=0.8, t_hi=0.8),
        # the 1,000 most balanced triangles
        dict(name="topk_cl1m", kind="topk", graph="cl", n=1000000, draws=10000000, gamma=2.1, dist="beta_half",
             order="sorted", K=1000, which=1),
    ]


DISTS = ("uniform", "beta_half", "mixture", "normal", "beta31", "beta13")
# largest graph (vertices) that is drawn for a kind
MOST_N = {"count": 1 << 22, "enumerate": 1 << 19, "train": 4000000, "worlds": 1 << 19, "host": 1 << 21,
          "aeo": 1 << 20, "sample": 1 << 20, "topk": 1 << 20}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("count", "count", "enumerate", "train", "worlds", "batch", "host", "aeo", "sample", "topk"))
    if kind == "batch":
        s_lo = _log_int(rng, 10, 200)
        return dict(kind=kind, graphs=_log_int(rng, 8, 900), s_lo=s_lo, s_hi=_log_int(rng, 2 * s_lo, 5000),
                    degree=rng.randint(8, 100), dist=rng.choice(DISTS), n_tau=rng.randint(1, 8), t_lo=0.55,
                    t_hi=round(rng.uniform(0.6, 0.98), 3))
    n = _log_int(rng, 700, MOST_N[kind])
    few = kind in ("enumerate", "aeo", "sample", "topk")  # answered at high thresholds: structures that have such triangles
    c = dict(kind=kind, graph=rng.choice(("cl", "rmat") if few else ("er", "cl", "rmat")), n=n,
             draws=int(n * rng.uniform(6.0, 15.0)), order=rng.choice(("sorted", "shuffled")),
             dist="real" if kind == "train" else rng.choice(DISTS[:3] if few else DISTS))
    if c["graph"] == "cl":
        c["gamma"] = round(rng.uniform(2.1, 2.8), 2)
    t_lo = round(rng.uniform(0.5, 0.8), 3)
    if kind in ("count", "host"):
        c.update(n_tau=_log_int(rng, 1, 64), t_lo=t_lo, t_hi=round(rng.uniform(t_lo, 0.99), 3), prune=rng.random() < 0.8)
    elif kind == "enumerate":
        c.update(t_lo=round(rng.uniform(0.9, 0.98), 3), which=rng.randint(1, 3), room=c["draws"])
    elif kind == "train":
        c.update(edges=int(c["draws"] * (0.4 if c["graph"] == "rmat" else 0.6)))
    elif kind == "worlds":
        c.update(worlds=64 * _log_int(rng, 1, 64))
    elif kind == "aeo":
        c.update(n_tau=_log_int(rng, 1, 64), t_lo=round(rng.uniform(0.6, 0.95), 3), t_hi=0.97)
    elif kind == "sample":
        c.update(of=rng.choice(("edges", "vertices")), samples=_log_int(rng, 100, 20000), n_tau=_log_int(rng, 1, 16),
                 t_lo=round(rng.uniform(0.6, 0.9), 3), t_hi=0.95)
    elif kind == "topk":
        c.update(K=_log_int(rng, 10, max(20, min(50000, n // 4))), which=rng.randint(1, 2))
    return c


# ------------------------------------------------------------------ inputs

def _rand(count, gen):
    return torch.rand(count, device="cuda", generator=gen)


def _probabilities(dist, m, gen):
    """P+ of m edges.  Beta laws with integer parameters are order statistics of uniforms."""
    if dist == "beta_half":  # Beta(1/2, 1/2) is the arcsine law
        return torch.sin(_rand(m, gen) * (math.pi / 2)) ** 2
    if dist == "mixture":    # 1/2 Beta(8, 2) + 1/2 Beta(2, 8): the second largest of nine, mirrored half the time
        first = _rand(m, gen)
        second = torch.zeros_like(first)
        for _ in range(8):
            x = _rand(m, gen)
            second = torch.maximum(second, torch.minimum(first, x))
            first = torch.maximum(first, x)
        return torch.where(_rand(m, gen) < 0.5, second, 1 - second)
    if dist == "normal":
        return (0.5 + 0.15 * torch.randn(m, device="cuda", generator=gen)).clamp_(0, 1)
    if dist == "beta31":
        return torch.maximum(torch.maximum(_rand(m, gen), _rand(m, gen)), _rand(m, gen))
    if dist == "beta13":
        return torch.minimum(torch.minimum(_rand(m, gen), _rand(m, gen)), _rand(m, gen))
    return _rand(m, gen)     # "uniform" and "real"


def _values(dist, m, gen):
    """k of m edges (int32), uniform ones over all of 0..65536."""
    if dist == "uniform":
        return torch.randint(0, ONE + 1, (m,), device="cuda", generator=gen, dtype=torch.int32)
    return torch.round(_probabilities(dist, m, gen) * ONE).clamp_(0, ONE).to(torch.int32)


def _endpoints(case, gen):
    n, draws = case["n"], case["draws"]
    if case["graph"] == "er":
        return (torch.randint(0, n, (draws,), device="cuda", generator=gen),
                torch.randint(0, n, (draws,), device="cuda", generator=gen))
    if case["graph"] == "cl":  # Chung-Lu: power-law weights, the mean kept after the cap
        mean, most = 2.0 * draws / n, min(50000.0, n / 4)
        base = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** (-1.0 / (case["gamma"] - 1.0))
        lo, hi = torch.zeros((), device="cuda", dtype=torch.float64), mean * n / base.sum() * 1e4
        for _ in range(60):
            mid = (lo + hi) / 2
            low = (base * mid).clamp_(max=most).mean() < mean
            lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
        cdf = torch.cumsum((base * hi).clamp_(max=most), 0)
        cdf = cdf / cdf[-1].clone()
        a, b = (torch.searchsorted(cdf, torch.rand(draws, device="cuda", dtype=torch.float64, generator=gen))
                for _ in range(2))
        return a.clamp_(max=n - 1), b.clamp_(max=n - 1)
    u = torch.zeros(draws, device="cuda", dtype=torch.int64)  # R-MAT (0.57, 0.19, 0.19, 0.05)
    v = torch.zeros_like(u)
    for _ in range(max(1, (n - 1).bit_length())):
        r = _rand(draws, gen)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    ok = (u < n) & (v < n)
    return u[ok], v[ok]


def _simple(a, b, n):
    """The distinct unordered pairs among (a, b), no self-loops, sorted."""
    ok = a != b
    a, b = a[ok], b[ok]
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    return key // n, key % n


def _graph(case, gen):
    """(src, dst) int32: sorted pairs, or in random order and orientation as they come from a file."""
    src, dst = _simple(*_endpoints(case, gen), case["n"])
    if src.numel() > case.get("edges", src.numel()):  # a random part of them: the same number for every seed
        at = torch.randperm(src.numel(), device="cuda", generator=gen)[: case["edges"]].sort().values
        src, dst = src[at], dst[at]
    if case["order"] == "shuffled":
        at = torch.randperm(src.numel(), device="cuda", generator=gen)
        flip = _rand(src.numel(), gen) < 0.5
        src, dst = src[at], dst[at]
        src, dst = torch.where(flip, dst, src), torch.where(flip, src, dst)
    return src.to(torch.int32), dst.to(torch.int32)


def _batch(case, gen, seed):
    """Disjoint graphs with log-uniform sizes: a centre joined to everyone and power-law pairs among the members."""
    r = np.random.default_rng(seed)
    sizes = np.rint(np.exp(r.uniform(math.log(case["s_lo"]), math.log(case["s_hi"]), case["graphs"]))).astype(np.int64)
    pairs = sizes * np.minimum(case["degree"], sizes // 4) // 2
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    s = torch.from_numpy(sizes).cuda()
    g = torch.repeat_interleave(torch.arange(case["graphs"], device="cuda"), torch.from_numpy(pairs).cuda())
    one = [off[g] + (s[g] * _rand(g.numel(), gen) ** 2).to(torch.int64) for _ in range(2)]
    a, b = (torch.minimum(x, off[g + 1] - 1) for x in one)
    n = int(sizes.sum())
    member = torch.arange(n, device="cuda")
    centre = torch.repeat_interleave(off[:-1], s)
    src, dst = _simple(torch.cat([a, centre]), torch.cat([b, member]), n)
    return n, off, src.to(torch.int32), dst.to(torch.int32)


def _taus(case):
    return np.linspace(case["t_lo"], case["t_hi"], case["n_tau"])


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "batch":
        n, off, src, dst = _batch(case, gen, seed)
    else:
        n, off = case["n"], None
        src, dst = _graph(case, gen)
    p = k = None
    if case["dist"] == "real":
        p = _probabilities("real", src.numel(), gen)
    else:
        k = _values(case["dist"], src.numel(), gen)
    more = {}
    if case["kind"] == "batch":  # the edges' ids in the graph the members come from
        more["key"] = torch.randint(0, 1 << 24, (src.numel(),), device="cuda", generator=gen, dtype=torch.int32)
    if case["kind"] == "sample":
        most = src.numel() if case["of"] == "edges" else n
        more["items"] = torch.randint(0, most, (case["samples"],), device="cuda", generator=gen, dtype=torch.int32)
    return dict(n=n, off=off, src=src, dst=dst, k=k, p=p, **more)


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    state = dict(case=case, seed=seed)
    if kind == "host":
        host = lambda t: t.cpu().numpy().view(np.uint32)  # noqa: E731
        state.update(n=x["n"], src=host(x["src"]), dst=host(x["dst"]), k=host(x["k"]))
    elif kind == "aeo":
        state.update(n=x["n"], src=x["src"], dst=x["dst"], k=x["k"])
    elif kind == "train":
        state.update(G=ubt.Graph(x["n"], x["src"], x["dst"], p=x["p"]), p=x["p"].requires_grad_(True))
    elif kind == "batch":
        state.update(G=ubt.Graph(x["n"], x["src"], x["dst"], k=x["k"], edge_key=x["key"], vertex_offsets=x["off"]))
    elif kind == "sample":
        state.update(G=ubt.Graph(x["n"], x["src"], x["dst"], k=x["k"], undirected=True, edge_index=True),
                     items=x["items"])
    else:
        state.update(G=ubt.Graph(x["n"], x["src"], x["dst"], k=x["k"]))
    return state


# ------------------------------------------------------------------ the calls

def _in_order(key, p_bal, room):
    """Records by (u, v, w) in buffers of `room` entries, as a program keeps them."""
    key, at = torch.sort(key)
    held = min(room, key.numel())
    uvw = torch.full((room,), -1, device="cuda", dtype=torch.int64)
    p = torch.zeros(room, device="cuda", dtype=torch.float64)
    uvw[:held], p[:held] = key[:held], p_bal[at[:held]]
    return {"uvw": uvw, "p_bal": p}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "count":
        bal, unbal = state["G"].count_threshold(_taus(case), prune=case["prune"])
        return {"bal": bal, "unbal": unbal}
    if kind == "enumerate":
        rec = state["G"].enumerate(case["t_lo"], which=case["which"])
        key = (rec["u"].astype(np.int64) << 42) | (rec["v"].astype(np.int64) << 21) | rec["w"]  # n <= 2^21
        return _in_order(torch.from_numpy(key).cuda(), torch.from_numpy(np.ascontiguousarray(rec["p_bal"])).cuda(),
                         case["room"])
    if kind == "topk":
        rec = state["G"].topk(case["K"], which=case["which"])
        return {"uvw": np.stack([rec["u"], rec["v"], rec["w"]]).astype(np.int64),
                "p_bal": np.ascontiguousarray(rec["p_bal"])}
    if kind == "train":
        p = state["p"]
        p.grad = None
        bal, unbal = ubt.expected_counts(state["G"], p)
        (bal - unbal).backward()
        return {"bal": bal.detach(), "unbal": unbal.detach(), "grad": p.grad}
    if kind == "worlds":
        counts, total = state["G"].sample_worlds(state["seed"], case["worlds"])
        return {"counts": counts, "total": total}
    if kind == "batch":
        counts, expect, worlds = state["G"].batch_query(_taus(case), seed=state["seed"])
        return {"counts": counts, "expect": expect, "worlds": worlds}
    if kind == "host":
        bal, unbal = ubt.count_host(state["n"], state["src"], state["dst"], state["k"], _taus(case),
                                    prune=case["prune"])
        return {"bal": bal, "unbal": unbal}
    if kind == "aeo":
        G = ubt.Graph(state["n"], state["src"], state["dst"], k=state["k"], undirected=True, edge_index=True)
        bal, unbal = G.count_aeo(_taus(case))
        return {"bal": bal, "unbal": unbal}
    call = state["G"].edge_local_counts if case["of"] == "edges" else state["G"].vertex_local_counts
    bal, unbal, estimate = call(state["items"], _taus(case))
    return {"bal": bal, "unbal": unbal, "estimate": estimate}


# ------------------------------------------------------------------ the work

# edges kept of the pairs drawn (self-loops and repeated pairs go), as the structures above give them
KEPT = {"er": 1.0, "cl": 0.91, "rmat": 0.95}


def work(case):
    """Bytes of one pass: the forward lists (8 per edge, 4 per vertex) read once and the answers written once;
    builds read the 12-byte edges and write the lists.  The arithmetic is integer: no flops."""
    kind = case["kind"]
    if kind == "batch":
        sizes = np.exp(np.linspace(math.log(case["s_lo"]), math.log(case["s_hi"]), 1000)).astype(np.int64)
        n = float(case["graphs"] * sizes.mean())
        m = float(case["graphs"] * (sizes * np.minimum(case["degree"], sizes // 4) // 2).mean() * 0.9 + n)
    else:
        n, m = case["n"], case.get("edges", KEPT[case["graph"]] * case["draws"])
    lists = 8.0 * m + 4.0 * n
    out = 16.0 * case.get("n_tau", 1) + 16.0 * case.get("room", 0)
    if kind == "train":       # forward and backward each read the lists; p is read, its gradient written
        return {"bytes": 2 * lists + 8.0 * m, "flops": 0.0}
    if kind == "worlds":      # a sign bit per edge and world is drawn, kept and read again
        return {"bytes": lists + 2.0 * m * case["worlds"] / 8 + 8.0 * case["worlds"], "flops": 0.0}
    if kind == "batch":       # lists, keys, one sign word per edge; per graph counts, two sums and 64 worlds
        return {"bytes": lists + 12.0 * m + case["graphs"] * (out + 16 + 512), "flops": 0.0}
    if kind == "host":        # the edges cross to the device, are read there, and the lists are written and read
        return {"bytes": 24.0 * m + 2 * lists + out, "flops": 0.0}
    if kind == "aeo":         # both directions of every edge are written and read, and the 64-byte index slots
        return {"bytes": 12.0 * m + 2 * (lists + 24.0 * m) + 64.0 * m + out, "flops": 0.0}
    if kind == "sample":      # the rows of a sample and of its neighbours, of average length
        row = 8.0 * 2 * m / n
        rows = 2 if case["of"] == "edges" else 1 + 2 * m / n
        return {"bytes": case["samples"] * (rows * row + 4 + out), "flops": 0.0}
    if kind == "topk":
        return {"bytes": lists + 24.0 * case["K"], "flops": 0.0}
    return {"bytes": lists + out, "flops": 0.0}


# ------------------------------------------------------------------ the same in 64 bits

MOST_WEDGES = 8e9  # more than this takes too long here


def _triangles(n, src, dst, chunk=1 << 26):
    """The edge indices (i, j, l) of every triangle, in pieces; None where the graph has too many wedges."""
    src, dst = src.long(), dst.long()
    m = src.numel()
    deg = torch.bincount(torch.cat([src, dst]), minlength=n)
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[torch.argsort(deg, stable=True)] = torch.arange(n, device="cuda")
    a, b = rank[src], rank[dst]
    key, edge = torch.sort(torch.minimum(a, b) * n + torch.maximum(a, b))
    u, v = key // n, key % n
    end = torch.cumsum(torch.bincount(u, minlength=n), 0)
    later = end[u] - 1 - torch.arange(m, device="cuda")
    upto = torch.cumsum(later, 0)
    if m == 0 or int(upto[-1]) > MOST_WEDGES:
        return None if m else iter(())

    def pieces():
        at, done = 0, 0
        while at < m:
            to = max(at + 1, int(torch.searchsorted(upto, done + chunk, right=True)))
            cnt = later[at:to]
            i = torch.repeat_interleave(torch.arange(at, to, device="cuda"), cnt)
            j = i + 1 + torch.arange(i.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            want = v[i] * n + v[j]
            l = torch.searchsorted(key, want).clamp_(max=m - 1)
            hit = key[l] == want
            yield edge[i[hit]], edge[j[hit]], edge[l[hit]]
            done, at = int(upto[to - 1]), to

    return pieces()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("count", "host", "aeo", "worlds"):
        return None  # whole numbers
    x = _inputs(case, seed)
    n, src, dst = x["n"], x["src"], x["dst"]
    m = src.numel()
    if kind == "train":
        s = 1 - 2 * x["p"].double()
        T, S, grad = 0, 0.0, torch.zeros(m, dtype=torch.float64, device="cuda")
        tri = _triangles(n, src, dst)
        if tri is None:
            return None
        for i, j, l in tri:
            T += i.numel()
            S += float((s[i] * s[j] * s[l]).sum())
            for e, f, g in ((i, j, l), (j, i, l), (l, i, j)):
                grad.index_add_(0, e, 2 * s[f] * s[g])
        both = torch.tensor([(T - S) / 2, (T + S) / 2], dtype=torch.float64)
        return {"bal": both[0], "unbal": both[1], "grad": grad}
    q = ONE // 2 - x["k"].long()  # 1 - 2 P+ = q / 2^15
    unit = 2.0 ** 45
    if kind == "enumerate":
        c = (2 * case["t_lo"] - 1) * unit
        keep = (q.abs().double() * 2.0 ** 30 >= c).nonzero().flatten()  # the others are in no such triangle
        src, dst, q = src[keep], dst[keep], q[keep]
    tri = _triangles(n, src, dst)
    if tri is None:
        return None
    if kind == "enumerate":
        keys, vals = [], []
        for i, j, l in tri:
            P = (q[i] * q[j] * q[l]).double()
            bal, unbal = P <= -c, P > c
            hit = (bal if case["which"] & 1 else unbal) | (unbal if case["which"] & 2 else bal)
            e = torch.stack([i[hit], j[hit], l[hit]])
            at = torch.sort(torch.cat([src[e], dst[e]]).long(), 0).values[::2]
            keys.append((at[0] << 42) | (at[1] << 21) | at[2])
            vals.append((unit - P[hit]) / (2 * unit))
        none = torch.zeros(0, dtype=torch.int64, device="cuda")
        kept = _in_order(torch.cat(keys + [none]), torch.cat(vals + [none.double()]), case["room"])
        return {"uvw": None, "p_bal": kept["p_bal"]}
    if kind == "topk":
        best = torch.zeros(0, dtype=torch.float64, device="cuda")
        for i, j, l in tri:
            best = torch.cat([best, (q[i] * q[j] * q[l]).double()])
            best = torch.topk(best, min(case["K"], best.numel()), largest=case["which"] == 2).values
        return {"uvw": None, "p_bal": (unit - best) / (2 * unit)}
    if kind == "batch":
        of = torch.searchsorted(x["off"], src.long(), right=True) - 1
        T, S = (torch.zeros(case["graphs"], dtype=torch.float64, device="cuda") for _ in range(2))
        for i, j, l in tri:
            P = (q[i] * q[j] * q[l]).double() / unit
            S.index_add_(0, of[i], P)
            T.index_add_(0, of[i], torch.ones_like(P))
        return {"counts": None, "expect": torch.stack([(T - S) / 2, (T + S) / 2], 1), "worlds": None}
    size, taus = (m if case["of"] == "edges" else n), _taus(case)
    local = torch.zeros(2, len(taus), size, dtype=torch.float64, device="cuda")
    for i, j, l in tri:
        P = (q[i] * q[j] * q[l]).double()
        if case["of"] == "edges":
            where = (i, j, l)
        else:
            e = torch.stack([i, j, l])
            where = torch.sort(torch.cat([src[e], dst[e]]).long(), 0).values[::2]
        for t, tau in enumerate(taus):
            c = (2 * float(tau) - 1) * unit
            for side, hit in ((0, P <= -c), (1, P > c)):
                for w in where:
                    local[side, t].index_add_(0, w, hit.double())
    return {"bal": None, "unbal": None, "estimate": local[:, :, x["items"].long()].mean(2) * (size / 3)}
