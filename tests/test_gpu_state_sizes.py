"""Populations on both sides of the size from which the device permutes them: put
in, read back, refused and carried through a checkpoint, in rows of bytes and bits."""
import numpy as np
import pytest

import oracle
from gpu_helpers import require_gpu
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,variant", [(128, 127, 0), (128, 128, 0), (128, 129, 0), (128, 511, 1), (128, 512, 1), (128, 513, 1),
                                         (128, 767, 1), (128, 768, 1), (128, 769, 1), (131, 33, 3), (4001, 17, 3),
                                         (1024, 255, 0), (1024, 257, 0), (1024, 255, 1), (1024, 257, 1)])
def test_both_sides_of_the_size_rule(tmp_path, n, R, variant):
    require_gpu()
    g = wl.gnm(n, 3 * n, seed=n)
    x = (np.random.default_rng(R).integers(0, 2, (R, n)) * 2 - 1).astype(np.int8)
    E = np.array([oracle.energy(g.rp, g.col, g.w, row) for row in x], np.int32)
    bad = x.copy()
    bad[-1, -1] = 0
    with B.Annealer.from_graph(g) as a:
        a.begin(wl.linear_betas(0.1, 1.0, 4), R, 1, 7, variant=variant)
        a.set_state(x, 1)
        for call in (lambda: a.set_state(bad, 1), lambda: a.energies(bad)):
            with pytest.raises(B.PaError) as e:
                call()
            assert e.value.code == B.PA_EINVAL
        got = a.state()
        np.testing.assert_array_equal(got[0], x)
        np.testing.assert_array_equal(got[1], E)
        np.testing.assert_array_equal(a.energies(x)[0], E)
        a.save(str(tmp_path / "ck.bin"))
        a.run(4)
        want = a.state()
    with B.Annealer.from_graph(g) as a:
        a.load(str(tmp_path / "ck.bin"))
        np.testing.assert_array_equal(a.state()[0], x)
        a.run(4)
        got = a.state()
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
