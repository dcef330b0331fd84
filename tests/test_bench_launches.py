"""The benchmark's count of the library's own kernels: by name on the CPU, and
on the GPU against queries whose kernels are known."""
import pytest

import bench


def test_own_kernels_by_name():
    names = ["void ubt::(anonymous namespace)::k_traverse<ubt::(anonymous namespace)::CountBins, 1>(ubt::TravArgs)",
             "ubt::(anonymous namespace)::k_keep_count(unsigned long const*, long)", "Memset (Device)",
             "Memcpy DtoH (Device -> Pinned)", "void at::native::vectorized_elementwise_kernel<4>(int)"]
    assert bench.own_kernels(names) == 2
    assert bench.own_kernels([]) == 0


@pytest.mark.gpu
def test_launches_of_a_query():
    import numpy as np
    import torch

    import synth
    from gpu_util import core_graph, require_gpu
    ubt = require_gpu()
    out = torch.empty(4, dtype=torch.int64, device="cuda")
    s, d = core_graph(3000, 30000, 300, 5)
    k = synth.k_uniform(s.size, 6)
    G = ubt.Graph(3000, s, d, k=k)
    assert bench.kernels_of(lambda: G.count_threshold_([0.6, 0.9], out, prune=False)) == 1
    old = ubt.get_tuning("block_bits")
    try:
        ubt.set_tuning("block_bits", 0)  # block tasks with hash tables: a kernel of their own
        H = ubt.Graph(3000, s, d, k=k)
    finally:
        ubt.set_tuning("block_bits", old)
    assert bench.kernels_of(lambda: H.count_threshold_([0.6, 0.9], out, prune=False)) == 2
    s, d = synth.rmat(16, 32, 0.57, 0.19, 0.19, 5)
    P = ubt.Graph(1 << 16, s, d, k=synth.quantise(synth.p_beta_mixture(s.size, 6)))
    # kept entries: counted, scanned, written, their number
    assert bench.kernels_of(lambda: P.count_threshold_([0.95, 1.0], out, prune=True)) == 5
