"""Populations and configurations that cross between vertex order on the host and
position order on the device: every row alignment, each layout's energies, the
graphs that have no word kernels, and inputs that must be refused."""
import numpy as np
import pytest

import oracle
from gpu_helpers import require_gpu
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _spins(R, n, seed):
    return (np.random.default_rng(seed).integers(0, 2, (R, n)) * 2 - 1).astype(np.int8)


def _energies(g, x):
    return np.array([oracle.energy(g.rp, g.col, g.w, row) for row in x], np.int32)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 16, 17, 31, 33, 63, 130])
@pytest.mark.parametrize("opts", [dict(), dict(variant=1), dict(variant=3), dict(field_bits=16)])
def test_set_and_get_state_at_every_alignment(n, opts):
    require_gpu()
    g = wl.gnm(n, min(n * (n - 1) // 2, 2 * n), seed=n)
    for R in (1, 5, 33):
        x = _spins(R, n, R)
        with B.Annealer.from_graph(g) as a:
            a.begin(np.array([0.5, 0.6]), R, 1, 3, **opts)
            a.set_state(x, 0)
            s, E = a.state()
            np.testing.assert_array_equal(s, x)
            np.testing.assert_array_equal(E, _energies(g, x))


@pytest.mark.parametrize("pos", [0, 7, 16, 32, -1])
@pytest.mark.parametrize("value", [0, 2, -2, 3, 127, -128])
def test_bad_spins_are_refused_and_change_nothing(pos, value):
    require_gpu()
    g = wl.gnm(37, 90, seed=1)
    x = _spins(3, 37, 1)
    bad = x.copy()
    bad.reshape(-1)[pos] = value
    with B.Annealer.from_graph(g) as a:
        a.begin(np.array([0.5]), 3, 1, 3)
        a.set_state(x, 0)
        for call in (lambda: a.set_state(bad, 0), lambda: a.energies(bad)):
            with pytest.raises(B.PaError) as e:
                call()
            assert e.value.code == B.PA_EINVAL
        s, E = a.state()
        np.testing.assert_array_equal(s, x)
        np.testing.assert_array_equal(E, _energies(g, x))


@pytest.mark.parametrize("R", [1, 31, 32, 33, 70])
@pytest.mark.parametrize("kind", ["signed", "dense", "big", "widest"])
def test_energies_of_configurations(R, kind):
    """16- and 32-bit slice rows, degrees above 127 and graphs beyond shared memory."""
    require_gpu()
    if kind == "signed":
        g = wl.torus(11, seed=3)
    elif kind == "dense":
        g = wl.gnp(300, 0.6, seed=4)
    elif kind == "big":
        g = wl.gnm(17001, 40000, seed=5)
    else:
        g = wl.gnm(60001, 70000, seed=6)
    x = _spins(R, g.n, R)
    with B.Annealer.from_graph(g) as a:
        E, cuts = a.energies(x)
    np.testing.assert_array_equal(E, _energies(g, x))
    W = oracle.total_weight(g.rp, g.col, g.w)
    np.testing.assert_array_equal(cuts, (W - E.astype(np.int64)) // 2)
