"""The chain between steps: the minimum a sweep leaves for the next step's weights
(every layout, non-local moves in between, a replaced population) and the
one-cluster resampling at all its shapes, with long runs of one parent."""
import numpy as np
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [255, 257, 512, 1025, 4097, 16385, 33000, 65536])
def test_resampling_shapes_and_long_runs(R):
    """A jump in beta leaves a few parents most of the slots."""
    require_gpu()
    g = wl.gnm(24, 60, seed=R)
    betas = np.array([0.0, 0.02, 1.5, 1.6])
    gpu = run_gpu(g, betas, R, 1, seed=R)
    orc = run_oracle(g, betas, R, 1, seed=R)
    assert orc.step_counts.max() > 8
    assert_parity(gpu, orc, g, R, 1)


@pytest.mark.parametrize("opts", [dict(), dict(variant=1), dict(variant=3), dict(field_bits=16), dict(field_bits=8)])
@pytest.mark.parametrize("nlm", [dict(), dict(nlm_period=2), dict(nlm_period=1, nlm_kind=1, nlm_block=5)])
def test_minimum_between_steps(opts, nlm):
    require_gpu()
    g = wl.gnm(150, 500, seed=2)
    betas = wl.linear_betas(0.1, 2.0, 7)
    gpu = run_gpu(g, betas, 41, 2, seed=4, **opts, **nlm)
    orc = run_oracle(g, betas, 41, 2, seed=4, **nlm)
    assert_parity(gpu, orc, g, 41, 2)


@pytest.mark.parametrize("opts", [dict(), dict(variant=1)])
def test_replaced_population_forgets_the_old_minimum(opts):
    """Steps run on another population leave nothing to a population put in its
    place, ahead of it or back in the schedule."""
    require_gpu()
    g = wl.gnm(150, 500, seed=2)
    betas = wl.linear_betas(0.1, 3.0, 9)
    x = (np.random.default_rng(1).integers(0, 2, (41, 150)) * 2 - 1).astype(np.int8)
    for ran, at in ((3, 3), (5, 2), (1, 6)):
        got = []
        for first in (ran, 0):
            with B.Annealer.from_graph(g) as a:
                a.begin(betas, 41, 2, 9, record_counts=1, **opts)
                if first:
                    a.run(first)
                a.set_state(x, at)
                a.run(9)
                a.sync()
                rec = a.step_stats(counts=True)
                got.append((a.state(), rec["emin"][at:], rec["A"][at:], rec["counts"][at:]))
        (s1, e1), m1, A1, c1 = got[0]
        (s2, e2), m2, A2, c2 = got[1]
        assert np.array_equal(s1, s2) and np.array_equal(e1, e2)
        assert np.array_equal(m1, m2) and np.array_equal(A1, A2) and np.array_equal(c1, c2)


ESS = dict(adaptive=1, rho=0.6, adapt_J=5, adapt_dbeta_max=0.25, beta_max=2.0)
ACC = dict(adaptive=2, adapt_J=4, adapt_dbeta_max=0.4, beta_max=3.0, acc_lo=0.12, acc_hi=0.3)


@pytest.mark.parametrize("opts", [dict(), dict(variant=1), dict(variant=3), dict(field_bits=16), dict(field_bits=8),
                                  dict(field_bits=7, threads_per_cta=128), ESS, dict(variant=3, **ESS), ACC,
                                  dict(reheat_after=4, reheat_back=2), dict(variant=1, nlm_period=3)])
@pytest.mark.parametrize("R", [70, 2500])
def test_many_short_steps(opts, R):
    """Steps of a few microseconds, each launched while the one before it ends."""
    require_gpu()
    g = wl.gnm(300, 900, seed=3)
    betas = None if "adaptive" in opts else wl.linear_betas(0.05, 3.0, 60)
    K = 80 if betas is None else None
    kw = {k: v for k, v in opts.items() if k not in ("variant", "field_bits", "threads_per_cta")}
    gpu = run_gpu(g, betas, R, 1, seed=R, K=K, **opts)
    orc = run_oracle(g, betas, R, 1, seed=R, K=K, **kw)
    assert_parity(gpu, orc, g, R, 1)
