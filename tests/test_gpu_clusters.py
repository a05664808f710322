"""Words spread over a cluster of CTAs: every counter width with and without signs,
and with everything that acts on a population between two sweeps, as the automatic
layout runs small populations of graphs with large colour classes. Each test makes
sure that a cluster ran."""
import numpy as np
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl
from test_gpu_msc_planes import _hub_graph

pytestmark = pytest.mark.gpu


def _ctas(g, R, **opts):
    with B.Annealer.from_graph(g) as a:
        a.begin(None if opts.get("adaptive") else np.array([0.5]), R, 1, 1, K=1, **opts)
        return a.sweep_shape()["ctas"]


@pytest.mark.parametrize("maxdeg", [7, 15, 31, 63, 127])
@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("n", [1100, 2200])
def test_counter_widths_in_clusters(maxdeg, signed, n):
    require_gpu()
    g = _hub_graph(n, maxdeg, n, 7 * maxdeg + signed, signed)
    assert g.maxdeg == maxdeg
    assert _ctas(g, 40, variant=3) >= 2
    betas = np.array([0.0, 0.05, 0.45, 1.0, 2.0, 3.6, 30.0])
    gpu = run_gpu(g, betas, 40, 2, seed=maxdeg, variant=3)
    orc = run_oracle(g, betas, 40, 2, seed=maxdeg)
    assert_parity(gpu, orc, g, 40, 2)


MOVES = [dict(nlm_period=2), dict(nlm_period=2, nlm_kind=1, nlm_block=9),
         dict(adaptive=1, rho=0.6, adapt_J=4, adapt_dbeta_max=0.25, beta_max=1.5, nlm_period=3),
         dict(adaptive=2, adapt_J=4, adapt_dbeta_max=0.4, beta_max=2.0, acc_lo=0.12, acc_hi=0.3),
         dict(reheat_after=3, reheat_back=2, nlm_period=4, nlm_kind=1, nlm_block=5)]


def _cases():
    return [wl.torus(70, seed=5), wl.gnm(5000, 7000, seed=6)]


@pytest.mark.parametrize("moves", MOVES)
@pytest.mark.parametrize("which", [0, 1])
def test_moves_and_schedules_on_clusters(which, moves):
    """The automatic layout, three words with 6 live replicas in the last."""
    require_gpu()
    g = _cases()[which]
    assert _ctas(g, 70, **moves) >= 2
    betas = None if "adaptive" in moves else wl.linear_betas(0.1, 2.5, 10)
    K = 24 if betas is None else None
    gpu = run_gpu(g, betas, 70, 2, seed=3, K=K, **moves)
    assert gpu["stats"]["variant"] == 3
    orc = run_oracle(g, betas, 70, 2, seed=3, K=K, **moves)
    assert_parity(gpu, orc, g, 70, 2)


@pytest.mark.parametrize("moves", [MOVES[0], MOVES[2]])
def test_checkpoint_of_a_cluster_run(tmp_path, moves):
    require_gpu()
    g = _cases()[0]
    betas = None if "adaptive" in moves else wl.linear_betas(0.1, 2.5, 10)
    K = 24 if betas is None else 10
    with B.Annealer.from_graph(g) as a:
        a.anneal(betas, 70, 2, 3, K=K, **moves)
        assert a.sweep_shape()["ctas"] >= 2
        want = a.state(), a.best_record(), a.step_stats()
    with B.Annealer.from_graph(g) as a:
        a.begin(betas, 70, 2, 3, K=K, **moves)
        a.run(4)
        a.save(str(tmp_path / "ck.bin"))
    with B.Annealer.from_graph(g) as a:
        a.load(str(tmp_path / "ck.bin"))
        assert a.sweep_shape()["ctas"] >= 2
        a.run(K)
        got = a.state(), a.best_record(), a.step_stats()
    np.testing.assert_array_equal(got[0][0], want[0][0])
    np.testing.assert_array_equal(got[0][1], want[0][1])
    assert got[1] == want[1]
    for key in ("beta", "emin", "A", "T", "o", "accepts", "sweep_emin", "nlm_pairs", "nlm_flips", "jsel"):
        np.testing.assert_array_equal(got[2][key], want[2][key], err_msg=key)
