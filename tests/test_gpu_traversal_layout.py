"""The arrays that the queries read, as the device holds them -- vertex
numbers, rows, pair words, pair partition, task lists and parts -- entry by
entry against a numpy construction of their definitions (include/ubt.h,
ubt_graph_export_traversal)."""
import numpy as np
import pytest

import synth
from gpu_util import core_graph, mixed_graph, require_gpu

pytestmark = pytest.mark.gpu

GIANT, HUB_HASH, HUB_BITS, MED_HASH, MED_BITS = range(5)
BITS_LEN, HEAVY_PAIRS, MERGE_DEGREE = 16384, 1 << 16, 32
PAIR_WORK, WORK_UNIT, PART_WORK, MAX_PARTS = 16, 8, 1 << 17, 1 << 15


@pytest.fixture(scope="module")
def ubt():
    return require_gpu()


def expected(ubt, n, s, d, k=None, p=None, offsets=None):
    """The same dictionary from the definitions; pairs sorted by (owner, word),
    tasks by class with every one's (log2 of work, owner, part, parts - 1)."""
    s, d, m = s.astype(np.int64), d.astype(np.int64), s.size
    deg = np.bincount(np.concatenate([s, d]), minlength=n)
    off = np.asarray([0, n] if offsets is None else offsets, dtype=np.int64)
    gid = np.searchsorted(off, np.arange(n), side="right") - 1
    vid = np.lexsort((-np.arange(n), -deg, gid))          # graph, degree descending, id descending
    num = np.empty(n, np.int64)
    num[vid] = np.arange(n)
    row, col = np.maximum(num[s], num[d]), np.minimum(num[s], num[d])
    eid = np.lexsort((col, row))
    row, col = row[eid], col[eid]
    length = np.bincount(row, minlength=n)
    row_ptr = np.concatenate([[0], np.cumsum(length)])
    if k is not None:
        val = 32768 - k.astype(np.int64)[eid]
        absq2 = np.abs(val) >> 1
    else:
        val = np.rint((1.0 - 2.0 * p.astype(np.float64)) * 2.0 ** 30).astype(np.int64)[eid]
        absq2 = np.zeros(m, np.int64)
    start = row_ptr[row]
    streamed = np.arange(m) - start
    word = (absq2.astype(np.uint64) << np.uint64(49)) | (streamed.astype(np.uint64) << np.uint64(32)) \
        | start.astype(np.uint64)
    npairs = np.bincount(col, minlength=n)
    order = np.lexsort((word, col))
    # tasks
    units = np.bincount(col, weights=(streamed + WORK_UNIT - 1) // WORK_UNIT, minlength=n).astype(np.int64)
    work = np.where(npairs > 0, WORK_UNIT * units + PAIR_WORK * npairs, 0)
    whole = int(streamed.sum()) + (WORK_UNIT + PAIR_WORK) * m
    hub = max(2, ubt.get_tuning("hub_threshold"))
    giant = max(hub, ubt.get_tuning("smem_table_max") // 4)
    limit = ubt.get_tuning("block_work")
    if limit == 1 << 14:
        limit = min(limit, max(2048, whole // 4096))
    part = max(min(PART_WORK, max(4096, whole // 2048)), whole // MAX_PARTS + 1)
    merge_from = n if offsets is not None else int((deg > MERGE_DEGREE).sum())
    x = np.arange(n)
    reach = x - off[gid]
    on = (length > 0) & (npairs > 0) & (x < merge_from)
    block = (length > hub) | (work > limit) | (npairs > HEAVY_PAIRS)
    bits = (reach <= ubt.get_tuning("block_bits")) & (length <= BITS_LEN)
    cls = np.where(length > giant, GIANT,
                   np.where(block, np.where(bits, HUB_BITS, HUB_HASH),
                            np.where(reach <= ubt.get_tuning("warp_bits"), MED_BITS, MED_HASH)))
    parts = np.where(cls <= HUB_BITS, np.minimum(work // part + 1, MAX_PARTS), 1)
    lg = np.where(work > 0, np.floor(np.log2(np.maximum(work, 1))), 0).astype(np.int64)
    tasks = [sorted((-int(lg[v]), int(v), i, int(parts[v]) - 1) for v in np.nonzero(on & (cls == c))[0]
                    for i in range(int(parts[v]))) for c in range(5)]
    pair_ptr = np.concatenate([[0], np.cumsum(npairs)])
    return {"vid": vid, "row_ptr": row_ptr, "col": col, "val": val, "eid": eid, "rowid": row, "pair_ptr": pair_ptr,
            "pairs": word[order], "tasks": tasks, "lg": lg,
            "merge_first": int(pair_ptr[merge_from]) if merge_from < n else m,
            "hub_vertices": int((on & (cls <= HUB_BITS)).sum())}


def check(ex, want):
    assert np.array_equal(ex["vid"], want["vid"])
    assert np.array_equal(ex["row_ptr"], want["row_ptr"])
    assert np.array_equal(ex["adj"] & np.uint64(0xFFFFFFFF), want["col"].astype(np.uint64))
    assert np.array_equal((ex["adj"] >> np.uint64(32)).astype(np.uint32).view(np.int32), want["val"])
    assert np.array_equal(ex["eid"], want["eid"])
    if ex["rowid"] is not None:
        assert np.array_equal(ex["rowid"], want["rowid"])
    assert np.array_equal(ex["pair_ptr"], want["pair_ptr"])
    owner = np.repeat(np.arange(want["vid"].size), np.diff(ex["pair_ptr"].astype(np.int64)))
    assert np.array_equal(ex["pairs"][np.lexsort((ex["pairs"], owner))], want["pairs"])
    assert ex["merge_first"] == want["merge_first"]
    at = 0
    for c in range(5):
        t = ex["tasks"][at: at + int(ex["task_sizes"][c])]
        at += t.size
        x, part, rest = [(t >> np.uint64(b)).astype(np.int64) & mask
                         for b, mask in ((0, 0xFFFFFFFF), (32, 0xFFFF), (48, 0xFFFF))]
        lg = want["lg"][x]
        assert np.all(np.diff(lg) <= 0), c  # heavier first
        assert sorted(zip((-lg).tolist(), x.tolist(), part.tolist(), rest.tolist())) == want["tasks"][c], c
    assert at == ex["tasks"].size


KNOBS = [{}, {"sort_smem_max": 64, "warp_sort_max": 128}, {"warp_sort_max": 512, "sort_smem_max": 256},
         {"warp_sort_max": 128, "sort_smem_max": 512}, {"block_work": 1}, {"block_work": 1 << 30},
         {"block_work": 1, "block_bits": 0}, {"block_bits": 90, "warp_bits": 33, "hub_threshold": 16},
         {"warp_bits": 0}, {"smem_table_max": 64, "hub_threshold": 8}, {"hub_threshold": 2, "block_work": 1 << 30}]


@pytest.mark.parametrize("knobs", KNOBS, ids=[",".join("%s=%d" % x for x in k.items()) or "default" for k in KNOBS])
@pytest.mark.parametrize("name", ["er", "mixed", "rmat14", "core"])
def test_arrays_of_a_graph(ubt, name, knobs):
    n, (s, d) = {"er": (5000, synth.er_graph(5000, 100000, 2)), "mixed": (3000, mixed_graph(3000, 30000, 5)),
                 "rmat14": (1 << 14, synth.rmat(14, 16, 0.57, 0.19, 0.19, 3)),
                 "core": (3000, core_graph(3000, 20000, 600, 15))}[name]
    k = synth.quantise(synth.p_beta(s.size, 0.5, 0.5, 4))
    p = synth.p_uniform_f32(s.size, 17)
    p[:5] = [0.0, 1.0, 0.5, 1e-30, 2.0 ** -24]
    old = {x: ubt.get_tuning(x) for x in knobs}
    try:
        for x, v in knobs.items():
            ubt.set_tuning(x, v)
        for values in ({"k": k}, {"p": p}):
            G = ubt.Graph(n, s, d, **values)
            want = expected(ubt, n, s, d, **values)
            check(G.export_traversal(), want)
            assert G.info()["hub_vertices"] == want["hub_vertices"]
    finally:
        for x, v in old.items():
            ubt.set_tuning(x, v)


@pytest.mark.parametrize("knobs", [{}, {"warp_bits": 0}, {"block_work": 1}])
def test_arrays_of_a_batch(ubt, knobs):
    n = 1 << 11
    ps, pd = synth.rmat(11, 16, 0.57, 0.19, 0.19, 11)
    eg = synth.ego_nets(n, ps, pd, 33, 3, 200, 13)
    k = synth.k_uniform(ps.size, 12)[eg["eid"]]
    nv = int(eg["v_off"][-1])
    old = {x: ubt.get_tuning(x) for x in knobs}
    try:
        for x, v in knobs.items():
            ubt.set_tuning(x, v)
        G = ubt.Graph(nv, eg["src"], eg["dst"], k=k, edge_key=eg["eid"], vertex_offsets=eg["v_off"])
        check(G.export_traversal(), expected(ubt, nv, eg["src"], eg["dst"], k=k, offsets=eg["v_off"]))
    finally:
        for x, v in old.items():
            ubt.set_tuning(x, v)


def test_the_check_sees_a_planted_mistake(ubt):
    """Mistakes put into the host copy: an entry out of order, a wrong length, a
    pair at another owner, a doubled task, a missing part, a wrong class."""
    s, d = core_graph(1100, 6000, 300, 9)
    k = synth.k_uniform(s.size, 10)
    G = ubt.Graph(1100, s, d, k=k)
    ex, want = G.export_traversal(), expected(ubt, 1100, s, d, k=k)
    check(ex, want)
    row = int(np.argmax(np.diff(ex["row_ptr"].astype(np.int64))))
    r0 = int(ex["row_ptr"][row])
    own = int(np.argmax(np.diff(ex["pair_ptr"].astype(np.int64)) > 1))
    p0 = int(ex["pair_ptr"][own])
    split = int(np.argmax((ex["tasks"] >> np.uint64(48)) > 0))
    assert ex["tasks"][split] >> np.uint64(48) > 0

    def plant(name, change):
        bad = dict(ex)
        bad[name] = ex[name].copy()
        change(bad[name])
        with pytest.raises(AssertionError):
            check(bad, want)

    def swap(a, i, j):
        a[[i, j]] = a[[j, i]]

    plant("adj", lambda a: swap(a, r0, r0 + 1))
    plant("eid", lambda a: swap(a, r0, r0 + 1))
    plant("rowid", lambda a: a.__setitem__(r0, row + 1))
    plant("pairs", lambda a: a.__setitem__(p0, a[p0] + np.uint64(1 << 32)))
    plant("pairs", lambda a: swap(a, p0, int(ex["pair_ptr"][own + 1])))
    plant("tasks", lambda a: a.__setitem__(split, a[split + 1]))
    plant("tasks", lambda a: a.__setitem__(split, a[split] - np.uint64(1 << 48)))
    plant("task_sizes", lambda a: a.__iadd__(np.array([0, 1, -1, 0, 0])))


@pytest.mark.parametrize("name", ["empty", "one", "core", "rmat15", "star"])
def test_edges_of_alg_2_keep_the_order_of_their_rows(ubt, name):
    """Every edge once, at the endpoint with the longer row (ties: the larger
    id), and an owner's edges in the order of its row."""
    n, (s, d) = {"empty": (7, (np.zeros(0, np.uint32), np.zeros(0, np.uint32))),
                 "one": (40, (np.array([3], np.uint32), np.array([39], np.uint32))),
                 "core": (3000, core_graph(3000, 20000, 600, 15)),
                 "rmat15": (1 << 15, synth.rmat(15, 16, 0.57, 0.19, 0.19, 3)),
                 "star": (70001, (np.zeros(70000, np.uint32), np.arange(1, 70001, dtype=np.uint32)))}[name]
    G = ubt.Graph(n, s, d, k=synth.k_uniform(s.size, 5), undirected=True)
    ex = G.export_undirected()
    up = ex["uptr"].astype(np.int64)
    deg = np.diff(up)
    row, col = np.repeat(np.arange(n), deg), ex["col"].astype(np.int64)
    own = (deg[row] > deg[col]) | ((deg[row] == deg[col]) & (row > col))
    pos = np.nonzero(own)[0]
    assert pos.size == s.size
    assert np.array_equal(ex["apair_ptr"], np.concatenate([[0], np.cumsum(np.bincount(row[pos], minlength=n))]))
    assert np.array_equal(ex["apair_pos"], pos) and np.array_equal(ex["apair_other"], col[pos])
