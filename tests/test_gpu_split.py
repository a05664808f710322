"""Sweeps whose last words run in CTA pairs beside the others: both launches have
the block size chosen for the whole, on a graph of which an SM holds two blocks as
on one of which it holds more, and the results are the oracle's."""
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,threads,K,opts", [(134, 512, 2, {}), (40, 256, 4, dict(nlm_period=2))])
def test_split_sweep_has_one_block_size(side, threads, K, opts):
    require_gpu()
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = wl.torus(side, seed=2)
    R = 32 * (sms + 3) - 5
    betas = wl.linear_betas(0.3, 1.8, K)
    with B.Annealer.from_graph(g) as a:
        a.begin(betas, R, 1, 4, variant=1, **opts)
        s = a.sweep_shape()
        assert (s["blocks"], s["tail_blocks"], s["tail_ctas"]) == (sms, 3, 2)
        assert s["threads"] == s["tail_threads"] == threads
        a.begin(betas, R, 1, 4, variant=1, msc_no_split=1, **opts)
        s = a.sweep_shape()
        assert (s["blocks"], s["tail_blocks"]) == (sms + 3, 0)
    gpu = run_gpu(g, betas, R, 1, seed=4, variant=1, **opts)
    orc = run_oracle(g, betas, R, 1, seed=4, **opts)
    assert_parity(gpu, orc, g, R, 1)
