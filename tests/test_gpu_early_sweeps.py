"""Sweeps placed while the resampling's CTAs still hold SMs: only where the blocks are
spread over the SMs as evenly as without them, with the oracle's results on both
sides of the rule."""
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("words,early", [(lambda sms: sms - 8, 1), (lambda sms: sms - 7, 0), (lambda sms: sms, 0),
                                         (lambda sms: 2 * sms - 16, 1), (lambda sms: 2 * sms - 15, 0)])
def test_words_beside_the_resampling(words, early):
    """Blocks of 256 threads, of which an SM holds four."""
    require_gpu()
    import torch

    g, R = wl.gnm(200, 500, seed=1), 32 * words(torch.cuda.get_device_properties(0).multi_processor_count)
    betas = wl.linear_betas(0.1, 1.5, 4)
    opts = dict(variant=1, msc_no_split=1)
    with B.Annealer.from_graph(g) as a:
        a.begin(betas, R, 1, 2, **opts)
        assert a.sweep_shape()["early"] == early
    gpu = run_gpu(g, betas, R, 1, seed=2, **opts)
    orc = run_oracle(g, betas, R, 1, seed=2)
    assert_parity(gpu, orc, g, R, 1)


def test_blocks_that_fill_their_slots_start_early():
    """1024 threads a block: no SM has room for a second one."""
    require_gpu()
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = wl.torus(60, seed=1)
    with B.Annealer.from_graph(g) as a:
        a.begin(wl.linear_betas(0.1, 1.0, 2), 4 * sms, 1, 2, variant=0)
        s = a.sweep_shape()
        assert (s["threads"], s["blocks"], s["early"]) == (1024, sms, 1)
