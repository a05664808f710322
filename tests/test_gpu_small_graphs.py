"""Parity of the small-graph kernel (layouts with fields, every colour class
within one round of the block) at the edges of its ranges: class sizes at its
limits, rows longer and shorter than a thread reads ahead, one to many blocks
per SM, both layouts, and the general kernels just beyond."""
import numpy as np
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _bipartite(a, b, m, seed, signed=True):
    """Two classes of a and b vertices with m random edges between them."""
    rng = np.random.default_rng(seed)
    pick = rng.choice(a * b, size=min(m, a * b), replace=False)
    i, j = pick // b, a + pick % b
    w = (rng.integers(0, 2, size=len(i)) * 2 - 1).astype(np.int8) if signed else None
    return wl.from_edges(a + b, i, j, w)


def _check(g, R, S, seed, betas, **opts):
    gpu = run_gpu(g, betas, R, S, seed, variant=0, **opts)
    orc = run_oracle(g, betas, R, S, seed)
    assert_parity(gpu, orc, g, R, S)


@pytest.mark.parametrize("a,b,m", [(1, 1, 1), (2, 3, 4), (128, 128, 3000), (129, 100, 2000), (256, 3, 300),
                                   (256, 256, 6000), (257, 8, 500)])
@pytest.mark.parametrize("field_bits", [0, 16])
def test_class_sizes(a, b, m, field_bits):
    require_gpu()
    g = _bipartite(a, b, m, a + b)
    _check(g, 9, 3, a, np.array([0.05, 0.3, 0.9, 2.2]), field_bits=field_bits)


@pytest.mark.parametrize("R", [1, 4, 6, 1300, 1900, 3100])
def test_blocks_per_sm(R):
    """One block, ragged last blocks, and the steps of the launch rule."""
    require_gpu()
    _check(wl.gnp(90, 0.2, seed=R), R, 2, R, np.array([0.1, 0.6, 1.5]))


@pytest.mark.parametrize("R", [5, 1000, 2000, 10000])
def test_long_rows_int16(R):
    """Degrees above 127 (int16 fields), signed: many units per thread."""
    require_gpu()
    g = wl.gnp(300, 0.5, seed=3)
    rng = np.random.default_rng(3)
    i, j, _ = g.edges()
    g = wl.from_edges(300, i, j, (rng.integers(0, 2, size=len(i)) * 2 - 1).astype(np.int8))
    assert g.maxdeg > 127
    _check(g, R, 1, R, np.array([0.02, 0.2]))


def test_general_int16_without_and_with_queue():
    """The int16 kernel with its queue, and on a graph that leaves no room for it."""
    require_gpu()
    _check(wl.gnm(3000, 9000, seed=1), 5, 2, 1, np.array([0.2, 1.0]), field_bits=16)
    _check(wl.gnm(18900, 40000, seed=2), 5, 1, 2, np.array([0.2, 1.0]), field_bits=16)
