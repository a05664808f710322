"""Kernels whose shared memory lies just below, at and above the 48 KB that a
launch may have without asking for more, static part included. A limit that one
graph raised lasts for the process, so every size runs in a process of its own."""
import os
import subprocess
import sys

import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A vertex of degree 130: no slice rows, so each configuration's row is held in
# shared memory beside the partial sums.
ENERGIES = """
import sys
import numpy as np
import oracle
from paper_2510_21105_gb300 import binding as B, workloads as wl
n = int(sys.argv[1])
rng = np.random.default_rng(n)
i = np.concatenate([np.zeros(130, np.int64), np.arange(131, n - 1)])
j = np.concatenate([np.arange(1, 131), np.arange(132, n)])
g = wl.from_edges(n, i, j, (rng.integers(0, 2, len(i)) * 2 - 1).astype(np.int8))
assert g.maxdeg == 130
x = (rng.integers(0, 2, (3, n)) * 2 - 1).astype(np.int8)
with B.Annealer.from_graph(g) as a:
    E, _ = a.energies(x)
np.testing.assert_array_equal(E, [oracle.energy(g.rp, g.col, g.w, row) for row in x])
"""

# Block moves hold the row, two bitsets and the block beside their sums.
BLOCKS = """
import sys
import numpy as np
import oracle
from paper_2510_21105_gb300 import binding as B, workloads as wl
n = int(sys.argv[1])
g = wl.gnm(n, n, seed=n)
betas = wl.linear_betas(0.2, 1.5, 3)
o = dict(nlm_period=1, nlm_kind=1, nlm_block=32)
with B.Annealer.from_graph(g) as a:
    a.anneal(betas, 33, 1, 3, **o)
    spins, E = a.state()
    rec = a.step_stats()
ref = oracle.anneal(g.rp, g.col, g.w, betas, R=33, S=1, seed=3, **o)
np.testing.assert_array_equal(spins, ref.spins)
np.testing.assert_array_equal(E, ref.E)
np.testing.assert_array_equal(rec["nlm_flips"], ref.step_nlm_flips)
"""


def _run(script, *args):
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", script, *map(str, args)], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("n", [48896, 48897, 49152, 49153])
def test_energies_of_rows_around_48_kb(n):
    require_gpu()
    _run(ENERGIES, n)


@pytest.mark.parametrize("n", [39152, 39153, 39216, 39217])
def test_block_moves_around_48_kb(n):
    require_gpu()
    _run(BLOCKS, n)
