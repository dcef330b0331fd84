"""Sign worlds in less memory than the largest pass takes: the same counts, in
smaller passes, from whatever workspace of the least size or more is given."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from gpu_util import core_graph, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ubt():
    ubt = require_gpu()
    old = ubt.get_tuning("world_words_per_pass")
    ubt.set_tuning("world_words_per_pass", 64)  # the default, whatever ran before
    yield ubt
    ubt.set_tuning("world_words_per_pass", old)


def run_in(ubt, G, W, nbytes):
    """ubt_sample_worlds with a workspace of nbytes: (status, counts)."""
    import torch
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    out = torch.full((W,), -1, dtype=torch.int64, device="cuda")
    st = ubt.lib().ubt_sample_worlds(G.handle, ctypes.c_uint64(21), W, ctypes.c_void_p(out.data_ptr()), None,
                                     ctypes.c_void_p(ws.data_ptr()), nbytes,
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return st, out.cpu().numpy()


@pytest.mark.parametrize("W", [64, 320, 1024, 4160])
def test_any_workspace_from_the_least_size_on(ubt, W):
    s, d = core_graph(400, 2500, 60, 9)
    k = synth.k_uniform(s.size, 10)
    G = ubt.Graph(400, s, d, k=k)
    words, m = W // 64, s.size
    least = 1
    while 2 * least <= min(8, words):
        least *= 2
    want = oracle.world_counts(400, s, d, k, 21, list(range(words)))
    most = G.sample_worlds_workspace(W)
    for w in (1, 2, 3, 8, 12, 16, 31, 64, 100):
        if w < least or m * w * 8 + 256 > 2 * most:
            continue
        st, got = run_in(ubt, G, W, m * w * 8 + 256)
        assert st == 0 and np.array_equal(got, want), w
    st, got = run_in(ubt, G, W, m * least * 8 + 255)
    assert st == -8 and (got == -1).all()
    assert G.guard() == 0


def test_where_the_largest_table_does_not_fit(ubt):
    """Where the allocator has no room for the largest pass's table, the call
    runs with a smaller one."""
    import torch
    s, d = core_graph(20000, 400000, 200, 5)
    k = synth.k_uniform(s.size, 6)
    G = ubt.Graph(20000, s, d, k=k)
    want, total = G.sample_worlds(seed=4, W=4096)
    assert G.sample_worlds_workspace(4096) > 64 * 8 * s.size
    torch.cuda.empty_cache()
    _, whole = torch.cuda.mem_get_info()
    try:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + 20 * 8 * s.size) / whole)
        got, t = G.sample_worlds(seed=4, W=4096)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert np.array_equal(got, want) and t == total


def test_the_size_follows_the_free_memory(ubt):
    """A table of more than 1 GiB is asked for only where the device has room."""
    import torch
    s, d = synth.er_graph(100000, 2300000, 5)
    G = ubt.Graph(100000, s, d, k=synth.k_uniform(s.size, 6))
    large = G.sample_worlds_workspace(4096)
    assert large > 1 << 30
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        free, _ = torch.cuda.mem_get_info()
        need = G.sample_worlds_workspace(4096)
        assert 8 * 8 * s.size < need < min(large, free)
        got, t = G.sample_worlds(seed=4, W=4096)
    finally:
        del fill
        torch.cuda.empty_cache()
    want, total = G.sample_worlds(seed=4, W=4096)
    assert np.array_equal(got, want) and t == total
