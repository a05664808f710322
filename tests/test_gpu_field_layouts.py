"""The int8 and int16 layouts' launch rule: threads by what an SM can hold of the
blocks, and the queue of accepted items only where rows are long against the class;
the oracle's results on every side of it."""
import numpy as np
import pytest

from gpu_helpers import assert_parity, require_gpu, run_gpu, run_oracle
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _hub(n, m, degree):
    i, j, _ = wl.gnm(n, m, seed=4).edges()
    e = np.array(sorted(set(zip(i.tolist(), j.tolist())) | {(0, k) for k in range(1, degree + 1)}))
    return wl.from_edges(n, e[:, 0], e[:, 1])


CASES = {
    # shared memory holds two blocks, five an SM to run: no more threads to win
    "torus int8": (lambda: wl.torus(100, seed=1), lambda sms: 20 * sms, dict(variant=0, field_bits=8), 512, 0),
    # short classes, many blocks: small ones
    "random int8": (lambda: wl.gnm(2000, 6000, seed=2), lambda sms: 36 * sms, dict(variant=0, field_bits=8), 128, 0),
    "random int16, few blocks": (lambda: wl.gnm(3000, 9000, seed=3), lambda sms: 21, dict(variant=0, field_bits=16), 512, 0),
    # a sparse graph that takes int16 fields for one vertex of degree 200
    "hub": (lambda: _hub(3000, 9000, 200), lambda sms: 12 * sms, dict(), 256, 0),
    "long rows int8": (lambda: wl.gnp(300, 0.2, seed=5), lambda sms: 30, dict(variant=0, field_bits=8), 512, 1),
    "long rows int16": (lambda: wl.gnp(400, 0.3, seed=6), lambda sms: 50, dict(replicas_per_cta=8), 512, 1),
}


@pytest.mark.parametrize("case", list(CASES))
def test_launch_rule(case):
    require_gpu()
    import torch

    graph, population, opts, threads, queue = CASES[case]
    g, R = graph(), population(torch.cuda.get_device_properties(0).multi_processor_count)
    betas = np.array([0.1, 0.9])
    with B.Annealer.from_graph(g) as a:
        a.begin(betas, R, 1, 6, **opts)
        s = a.sweep_shape()
    assert s["variant"] == 0 and not s["small_graph"]
    assert (s["threads"], s["row_queue"]) == (threads, queue)
    gpu = run_gpu(g, betas, R, 1, seed=6, **opts)
    orc = run_oracle(g, betas, R, 1, seed=6)
    assert_parity(gpu, orc, g, R, 1)
