"""A build whose pairs nearly all have one owner takes about as long as one
whose owners are all different."""
import time

import numpy as np
import pytest

import synth
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ubt():
    return require_gpu()


def best_build(ubt, n, s, d):
    import torch
    dev = [torch.from_numpy(np.asarray(x, np.uint32).view(np.int32)).cuda()
           for x in (s, d, synth.k_uniform(len(s), 5))]
    best = float("inf")
    for _ in range(6):
        torch.cuda.synchronize()
        t = time.perf_counter()
        G = ubt.Graph(n, dev[0], dev[1], k=dev[2])
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
        G.close()
    return best


def test_star_against_path(ubt):
    m = 8000000
    path = best_build(ubt, m + 1, np.arange(m), 1 + np.arange(m))
    star = best_build(ubt, m + 1, np.zeros(m), 1 + np.arange(m))
    assert star < 1.55 * path, (star, path)
