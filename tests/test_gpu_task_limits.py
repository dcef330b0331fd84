"""What the sizes a graph reports and the limits a tuning sets mean, and
launches whose shared memory is near the device's limit."""
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


class knobs:
    def __init__(self, ubt, **values):
        self.ubt, self.values = ubt, values

    def __enter__(self):
        self.old = {k: self.ubt.get_tuning(k) for k in self.values}
        for k, v in self.values.items():
            self.ubt.set_tuning(k, v)

    def __exit__(self, *exc):
        for k, v in self.old.items():
            self.ubt.set_tuning(k, v)


def clique(n):
    a, b = np.triu_indices(n, 1)
    return a.astype(np.uint32), b.astype(np.uint32)


def test_hub_vertices_counts_vertices(ubt):
    """In a 400-clique with block_work 1, every vertex with a list and a pair
    (all but the first and the last) is handled by whole blocks, most in
    several parts, and is one vertex."""
    s, d = clique(400)
    with knobs(ubt, block_work=1):
        G = ubt.Graph(400, s, d, k=synth.k_uniform(s.size, 1))
    assert G.info()["hub_vertices"] == 398


@pytest.mark.parametrize("block_work", [1 << 16, 1 << 20, 1 << 30])
def test_block_work_is_a_plain_limit(ubt, block_work):
    """A limit that no owner of a 120-clique reaches leaves no block tasks."""
    s, d = clique(120)
    k = synth.k_uniform(s.size, 2)
    with knobs(ubt, block_work=block_work):
        G = ubt.Graph(120, s, d, k=k)
    assert G.info()["hub_vertices"] == 0
    want = oracle.count_threshold(120, s, d, k, [0.6, 0.9])
    got = G.count_threshold([0.6, 0.9])
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_default_block_work_spreads_small_graphs(ubt):
    """The default limit is lowered for a small graph, so that no warp task is
    the whole query."""
    s, d = clique(120)
    assert ubt.Graph(120, s, d, k=synth.k_uniform(s.size, 2)).info()["hub_vertices"] > 0


def test_a_refused_launch_leaves_no_error_behind(ubt):
    """A tuning whose tables no block has the shared memory for is refused; the
    calls after it are not."""
    n = 9000
    s, d = core_graph(n, 300000, 4200, 3)
    k = synth.k_uniform(s.size, 4)
    with knobs(ubt, hub_threshold=4096, warp_bits=0, block_work=1 << 40):
        G = ubt.Graph(n, s, d, k=k)
        with pytest.raises(ubt.UbtError):
            G.sample_worlds(seed=5, W=64)
    w, total = ubt.Graph(n, s, d, k=k).sample_worlds(seed=5, W=64)
    assert total == int(w.sum())


def test_a_shape_near_the_limit_stays_allowed(ubt):
    """A launch with 226.4 KB of dynamic shared memory (a bitmap range of 65,536
    and a list of 3,850 entries a warp, eight warps) runs again after a smaller
    launch of the same kernel."""
    core, n = 3900, 70000
    s, d = clique(core)
    T = math.comb(core, 3)
    with knobs(ubt, hub_threshold=3850, warp_bits=65536, block_work=1 << 40, count_visitor=1):
        G = ubt.Graph(n, s, d, k=synth.k_uniform(s.size, 6))
        small_s, small_d = clique(80)
        S = ubt.Graph(80, small_s, small_d, k=synth.k_uniform(small_s.size, 7))
        first = G.count_threshold([0.5], prune=False)
        b, u = S.count_threshold([0.5], prune=False)
        assert b[0] + u[0] == math.comb(80, 3)
        again = G.count_threshold([0.5], prune=False)
    assert first[0][0] + first[1][0] == T
    assert again[0][0] == first[0][0] and again[1][0] == first[1][0]


@pytest.mark.parametrize("hub_threshold,warp_threads", [(1024, 64), (1024, 96), (1024, 128), (2048, 64)])
def test_worlds_with_large_warp_tables(ubt, hub_threshold, warp_threads):
    """Warp tables that leave no room for the block size the sign worlds prefer:
    smaller blocks, not a refusal."""
    n = 40000
    s, d = core_graph(n, 1200000, 600, 3)
    k = synth.k_uniform(s.size, 4)
    want, total = ubt.Graph(n, s, d, k=k).sample_worlds(seed=5, W=128)
    with knobs(ubt, hub_threshold=hub_threshold, warp_threads=warp_threads, warp_bits=0):
        G = ubt.Graph(n, s, d, k=k)
        got, t = G.sample_worlds(seed=5, W=128)
    assert np.array_equal(got, want) and t == total and G.guard() == 0
