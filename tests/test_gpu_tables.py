"""The traversal's tables and task classes: bitmaps and hash tables, warp and
block tasks, owners split into several block tasks, pruned edges written out
first.  Every way of choosing among them answers as the oracle does: counts,
records and exact sums are whole numbers or exact doubles, so the comparison
is exact; REAL expected counts within 1e-9 relative and gradients within the
floor of test_gpu_parity."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import core_graph, grad_report, mixed_graph, require_gpu, sort_records

pytestmark = pytest.mark.gpu

TAUS = [0.5, 0.55, 0.6, 0.75, 0.9, 0.99, 1.0]
# bitmap range of block tasks / of warp tasks; 0 keeps the hash tables, 33 cuts
# between the two inside the graph
KNOBS = [{}, {"block_bits": 0}, {"warp_bits": 0}, {"block_bits": 0, "warp_bits": 0}, {"warp_bits": 33},
         {"block_bits": 700, "warp_bits": 300, "hub_threshold": 16}, {"hub_threshold": 2, "block_work": 1},
         {"block_work": 1, "block_bits": 0}, {"warp_threads": 64, "hub_threshold": 8, "small_batch": 7}]


@pytest.fixture(scope="module")
def ubt():
    return require_gpu()


def graphs():
    s, d = mixed_graph(3000, 30000, 5)
    yield "mixed", 3000, s, d
    s, d = synth.rmat(13, 24, 0.57, 0.19, 0.19, 7)   # owners with enough work for several block tasks
    yield "rmat13", 1 << 13, s, d
    s, d = core_graph(1100, 4000, 160, 9)            # lists of 0..159 entries, ends of bitmap words
    yield "core", 1100, s, d


@pytest.mark.parametrize("knobs", KNOBS, ids=[",".join("%s=%d" % x for x in k.items()) or "default" for k in KNOBS])
@pytest.mark.parametrize("case", list(graphs()), ids=lambda c: c[0])
def test_tables_and_task_classes(ubt, case, knobs):
    name, n, s, d = case
    k = synth.quantise(synth.p_beta(s.size, 0.5, 0.5, 4))
    old = {x: ubt.get_tuning(x) for x in knobs}
    try:
        for x, v in knobs.items():
            ubt.set_tuning(x, v)
        G = ubt.Graph(n, s, d, k=k)
        ob, ou = oracle.count_threshold(n, s, d, k, TAUS)
        for prune in (0, 1):
            gb, gu = G.count_threshold(TAUS, prune=prune)
            assert np.array_equal(gb, ob) and np.array_equal(gu, ou), prune
        for t in (0.9, 0.99):
            ouvw, ocls, opb = oracle.enumerate_records(n, s, d, k, t, 3)
            uvw, cls, pb = sort_records(G.enumerate(t, 3))
            assert np.array_equal(uvw, ouvw) and np.array_equal(cls, ocls) and np.array_equal(pb, opb), t
        T, S = oracle.expected_fixed(n, s, d, k)
        _, _, T2, sumP = G.expected_counts(with_exact=True)
        assert T2 == T and S == T * (1 << 47) - 4 * sumP
        w, tot = G.sample_worlds(seed=3, W=128)
        assert np.array_equal(w, oracle.world_counts(n, s, d, k, 3, [0, 1])) and tot == int(w.sum())
        assert G.guard() == 0
        p = synth.p_uniform_f32(s.size, 17)
        import torch
        R = ubt.Graph(n, s, d, p=p)
        eb, eu = R.expected_counts()
        want, _, _ = oracle.expected_real(n, s, d, p)
        assert abs(eb - want) <= 1e-9 * max(1.0, want)
        grad = torch.empty(s.size, dtype=torch.float32, device="cuda")
        R.expected_counts_backward_(torch.tensor([1.0, 0.0], dtype=torch.float64, device="cuda"), grad)
        og, gabs = oracle.grad_real(n, s, d, p, with_abs=True)
        ok, _, _ = grad_report(grad.cpu().numpy().astype(np.float64), og, gabs)
        assert ok.all()
        assert R.guard() == 0
    finally:
        for x, v in old.items():
            ubt.set_tuning(x, v)


@pytest.mark.parametrize("t", [0.51, 0.7, 0.86, 0.95, 1.0])
def test_kept_edges_written_first(ubt, t):
    """A graph with enough probes that a pruned query writes the kept edges out
    first: counts of the levels where few, some and nearly all edges go."""
    n = 1 << 15
    s, d = synth.rmat(15, 24, 0.57, 0.19, 0.19, 5)
    k = synth.quantise(synth.p_beta_mixture(s.size, 6))
    k[::97] = 0
    k[1::97] = 65536
    G = ubt.Graph(n, s, d, k=k)
    want = oracle.count_threshold(n, s, d, k, [t])
    got = G.count_threshold([t], prune=True)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    rec = G.enumerate(t, 3) if t > 0.8 else None
    if rec is not None:
        assert rec.size == int(want[0][0]) + int(want[1][0])
    assert G.guard() == 0


@pytest.mark.parametrize("warp_bits", [0, 16384])
def test_batch_with_either_table(ubt, warp_bits):
    """Graphs of a batch at unaligned first vertices, with bitmaps and hash tables."""
    n = 1 << 11
    ps, pd = synth.rmat(11, 16, 0.57, 0.19, 0.19, 11)
    pk = synth.k_uniform(ps.size, 12)
    eg = synth.ego_nets(n, ps, pd, 33, 3, 200, 13)
    k = pk[eg["eid"]]
    old = ubt.get_tuning("warp_bits")
    try:
        ubt.set_tuning("warp_bits", warp_bits)
        G = ubt.Graph(int(eg["v_off"][-1]), eg["src"], eg["dst"], k=k, edge_key=eg["eid"], vertex_offsets=eg["v_off"])
    finally:
        ubt.set_tuning("warp_bits", old)
    counts, expect, worlds = G.batch_query([0.6, 0.9], seed=5)
    for gi in range(33):
        v0, v1 = int(eg["v_off"][gi]), int(eg["v_off"][gi + 1])
        e0, e1 = int(eg["e_off"][gi]), int(eg["e_off"][gi + 1])
        ls, ld, lk = eg["src"][e0:e1] - v0, eg["dst"][e0:e1] - v0, k[e0:e1]
        ob, ou = oracle.count_threshold(v1 - v0, ls, ld, lk, [0.6, 0.9])
        assert np.array_equal(counts[gi, 0], ob) and np.array_equal(counts[gi, 1], ou), gi
        T, S = oracle.expected_fixed(v1 - v0, ls, ld, lk)
        assert abs(expect[gi, 0] - S / float(1 << 48)) <= 1e-12 * max(1.0, T), gi
        assert np.array_equal(worlds[gi], oracle.world_counts(v1 - v0, ls, ld, lk, 5, [0], ekey=eg["eid"][e0:e1])), gi
    assert G.guard() == 0


@pytest.mark.parametrize("W", [64, 192, 448, 640, 3008, 4160])
def test_worlds_in_passes_of_every_size(ubt, W):
    """World counts whose words do not divide into passes of one size: last
    passes of other sizes, and with words to spare, under every largest pass."""
    s, d = core_graph(400, 2500, 60, 9)
    k = synth.k_uniform(s.size, 10)
    k[:50], k[50:100] = 0, 65536
    want = oracle.world_counts(400, s, d, k, 21, list(range(W // 64)))
    G = ubt.Graph(400, s, d, k=k)
    old = ubt.get_tuning("world_words_per_pass")
    try:
        for wpp in (1, 2, 8, 16, 64):
            ubt.set_tuning("world_words_per_pass", wpp)
            got, tot = G.sample_worlds(seed=21, W=W)
            assert np.array_equal(got, want) and tot == int(want.sum()), wpp
    finally:
        ubt.set_tuning("world_words_per_pass", old)
    assert G.guard() == 0


@pytest.mark.parametrize("smem_max", [64, 256, 4096])
@pytest.mark.parametrize("deg", [63, 64, 65, 257, 1030, 4095, 4097, 9000])
def test_undirected_rows_of_every_length(ubt, deg, smem_max):
    """A star of `deg` leaves and edges among them: a row at and around the
    lengths where its sort changes (registers, one block, runs merged in an
    odd or even number of rounds), with equal |q| (ties go by neighbour)."""
    n = deg + 200
    r = synth.rng(deg)
    leaves = r.choice(n - 1, size=deg, replace=False) + 1
    e = r.integers(1, n, size=(3000, 2))
    a = np.concatenate([np.zeros(deg, np.int64), e[:, 0]])
    b = np.concatenate([leaves, e[:, 1]])
    key = np.unique(np.minimum(a, b) * n + np.maximum(a, b))
    key = key[key // n != key % n]
    s, d = synth.random_orientation((key // n).astype(np.uint32), (key % n).astype(np.uint32), 3)
    k = (synth.k_uniform(s.size, 4) >> 12 << 12).astype(np.uint32)
    old = ubt.get_tuning("sort_smem_max"), ubt.get_tuning("warp_sort_max")
    try:
        ubt.set_tuning("warp_sort_max", 128)
        ubt.set_tuning("sort_smem_max", smem_max)
        G = ubt.Graph(n, s, d, k=k, undirected=True, edge_index=True)
    finally:
        ubt.set_tuning("sort_smem_max", old[0])
        ubt.set_tuning("warp_sort_max", old[1])
    ex = G.export_undirected()
    up = ex["uptr"].astype(np.int64)
    row = np.repeat(np.arange(n), np.diff(up))
    val, col, mir = ex["val"].astype(np.int64), ex["col"].astype(np.int64), ex["mirror"].astype(np.int64)
    key = (32768 - np.abs(val)) * (1 << 32) + col
    same = row[1:] == row[:-1]
    assert np.all(key[1:][same] > key[:-1][same])
    assert np.array_equal(val, 32768 - k.astype(np.int64)[ex["eid"]])
    assert np.array_equal(mir[mir], np.arange(2 * s.size)) and np.array_equal(row[mir], col)
    want = oracle.count_threshold(n, s, d, k, [0.55, 0.8])
    got = G.count_aeo([0.55, 0.8])
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert G.guard() == 0


@pytest.mark.parametrize("core,taus", [(640, [0.6, 0.95]), (1100, [0.5, 0.8])])
def test_edge_and_vertex_samples_of_long_rows_with_the_index(ubt, core, taus):
    """Samples looked up in the edge index by one warp (rows up to 512 entries of
    an edge, 32 of a vertex) or by many (longer rows, queued; rows of more than
    1,024 entries in a part of the queue kept for them): both sides of each
    limit, more samples than either part of the queue holds, repeats."""
    n = core + 900
    s, d = core_graph(n, 6000, core, 11)
    k = synth.k_uniform(s.size, 12)
    eb, eu, vb, vu = oracle.local_counts(n, s, d, k, taus)
    G = ubt.Graph(n, s, d, k=k, undirected=True, edge_index=True)
    es = synth.rng(13).integers(0, s.size, size=9000).astype(np.uint32)
    gb, gu, _ = G.edge_local_counts(es, taus)
    assert np.array_equal(gb, eb[es]) and np.array_equal(gu, eu[es])
    vs = synth.rng(14).integers(0, n, size=7000).astype(np.uint32)
    gb, gu, _ = G.vertex_local_counts(vs, taus)
    assert np.array_equal(gb, vb[vs]) and np.array_equal(gu, vu[vs])
    assert G.guard() == 0
