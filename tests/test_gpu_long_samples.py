"""Local counts of more long samples than the queue of the split launch holds:
the ones left over are counted by whole blocks, and count the same."""
import math

import numpy as np
import pytest

import oracle
import synth
from gpu_util import core_graph, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ubt():
    return require_gpu()


def clique_and_star(core, leaves):
    """A clique on `core` vertices and a star whose centre is vertex `core`."""
    a, b = np.triu_indices(core, 1)
    s = np.concatenate([a, np.full(leaves, core)]).astype(np.uint32)
    d = np.concatenate([b, core + 1 + np.arange(leaves)]).astype(np.uint32)
    return core + 1 + leaves, s, d


def test_a_hub_behind_a_full_queue_is_not_left_to_one_warp(ubt):
    """20,000 samples of a star's centre (1,025 entries, no triangle) fill the
    queue; the vertex of a 2,400-clique that comes last takes well under the
    time that one warp takes for it alone."""
    import torch
    core = 2400
    n, s, d = clique_and_star(core, 1025)
    G = ubt.Graph(n, s, d, k=synth.k_uniform(s.size, 3), undirected=True, edge_index=True)
    items = np.full(20001, core, np.uint32)
    items[-1] = 7

    def timed(x):
        t = torch.from_numpy(x.view(np.int32)).cuda()
        best = math.inf
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            out = G.vertex_local_counts(t, [0.5])
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best, out

    old = ubt.get_tuning("vertex_split")
    try:
        ubt.set_tuning("vertex_split", 1 << 32)  # no sample is queued: one warp each
        alone, (b1, u1, _) = timed(items[-1:])
    finally:
        ubt.set_tuning("vertex_split", old)
    behind, (b2, u2, _) = timed(items)
    assert b1[0, 0] + u1[0, 0] == math.comb(core - 1, 2)
    assert b2[-1, 0] == b1[0, 0] and u2[-1, 0] == u1[0, 0]
    assert not b2[:-1].any() and not u2[:-1].any()
    assert G.guard() == 0
    assert behind < 0.5 * alone, (behind, alone)


@pytest.mark.parametrize("taus", [[0.5], [0.8, 0.6, 0.95]])
@pytest.mark.parametrize("split", [32, 300, 1050])
def test_more_long_samples_than_the_queue_holds(ubt, split, taus):
    """Every sample's counts, with both parts of the queue full, the rest above
    and below the length that whole blocks take."""
    core, n = 1100, 2600
    s, d = core_graph(n, 30000, core, 11)
    k = synth.k_uniform(s.size, 12)
    eb, eu, vb, vu = oracle.local_counts(n, s, d, k, taus)
    G = ubt.Graph(n, s, d, k=k, undirected=True, edge_index=True)
    vs = synth.rng(14).integers(0, n, size=6000).astype(np.uint32)
    es = synth.rng(15).integers(0, s.size, size=8000).astype(np.uint32)
    old = ubt.get_tuning("vertex_split")
    try:
        ubt.set_tuning("vertex_split", split)
        gb, gu, est = G.vertex_local_counts(vs, taus)
        assert np.array_equal(gb, vb[vs]) and np.array_equal(gu, vu[vs])
        assert np.allclose(est[0], n / 3.0 * gb.mean(axis=0), rtol=1e-12)
        gb, gu, _ = G.edge_local_counts(es, taus)
        assert np.array_equal(gb, eb[es]) and np.array_equal(gu, eu[es])
    finally:
        ubt.set_tuning("vertex_split", old)
    assert G.guard() == 0
