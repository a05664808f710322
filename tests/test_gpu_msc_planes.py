"""Parity of the bit-sliced multi-spin-coded item at the edges of its ranges:
counter widths (largest degree just below and at a power of two), thresholds
from all-ones to none with a top byte, both row encodings, short tie queues."""
import numpy as np
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _hub_graph(n, maxdeg, m, seed, signed):
    """m random edges plus a hub of exactly maxdeg neighbours that no other
    vertex's degree exceeds."""
    rng = np.random.default_rng(seed)
    deg = np.zeros(n, np.int64)
    edges = {(0, j) for j in range(1, maxdeg + 1)}
    deg[0] = maxdeg
    deg[1:maxdeg + 1] = 1
    while len(edges) < m + maxdeg:
        a, b = sorted(int(v) for v in rng.integers(1, n, size=2))
        if a != b and (a, b) not in edges and deg[a] < maxdeg and deg[b] < maxdeg:
            edges.add((a, b))
            deg[[a, b]] += 1
    i, j = np.array(sorted(edges)).T
    w = (rng.integers(0, 2, size=len(i)) * 2 - 1).astype(np.int8) if signed else None
    return wl.from_edges(n, i, j, w)


@pytest.mark.parametrize("maxdeg", [2, 7, 8, 15, 16, 31, 32, 63, 64, 127])
@pytest.mark.parametrize("signed", [False, True])
def test_counter_widths(maxdeg, signed):
    """Every step draws from another regime: beta = 0 (all thresholds all-ones),
    many levels, a few, none with a top byte, all zero."""
    require_gpu()
    n = max(200, 3 * maxdeg)
    g = _hub_graph(n, maxdeg, n * min(maxdeg, 12) // 4, 7 * maxdeg + signed, signed)
    assert g.maxdeg == maxdeg
    betas = np.array([0.0, 0.01, 0.05, 0.2, 0.45, 0.7, 1.0, 1.4, 2.0, 2.8, 3.6, 6.0, 30.0])
    for variant in (1, 3):
        gpu = run_gpu(g, betas, 40, 3, seed=maxdeg, variant=variant)
        orc = run_oracle(g, betas, 40, 3, seed=maxdeg)
        assert_parity(gpu, orc, g, 40, 3)


@pytest.mark.parametrize("n,maxdeg,m", [(16384, 9, 20000), (16385, 33, 20000), (57000, 127, 40000)])
def test_row_encodings_and_short_queues(n, maxdeg, m):
    """The largest graph with 16-bit row entries, the smallest with 32-bit ones,
    and one that leaves the tie queues four entries per warp."""
    require_gpu()
    g = _hub_graph(n, maxdeg, m, n, True)
    betas = np.array([0.02, 0.6, 2.0])
    gpu = run_gpu(g, betas, 33, 1, seed=5, variant=1)
    orc = run_oracle(g, betas, 33, 1, seed=5)
    assert_parity(gpu, orc, g, 33, 1)


@pytest.mark.parametrize("n,R,variant", [
    (8001, 33, 3), (8001, 700, 3), (8001, 1300, 3), (8001, 2500, 3), (8001, 5000, 3),   # 8, 4, 2, 1 CTAs per word; pairs past one word per SM
    (8001, 33, 1), (250, 40, 1),                                                        # one CTA: 512 threads, and 256 for a short class
    (18000, 4870, 1), (40000, 33, 3)])                                                  # two CTAs, one CTA in an SM's shared memory
def test_threads_and_clusters(n, R, variant):
    """Each block size and cluster size of the launch rule."""
    require_gpu()
    g = _hub_graph(n, 9, 2 * n, n, True)
    betas = np.array([0.3, 1.5])
    gpu = run_gpu(g, betas, R, 1, seed=R, variant=variant)
    orc = run_oracle(g, betas, R, 1, seed=R)
    assert_parity(gpu, orc, g, R, 1)
