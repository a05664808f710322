"""What a served request is charged against the memory budget: the rows of its
layout, one bit a spin where 32 replicas share a word."""
import time

import pytest

from gpu_helpers import require_gpu
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

G, R, K = (2000, 12000), 8192, 12


def _running(srv, rid):
    t_end = time.time() + 30
    while srv.poll(rid) == 0 and time.time() < t_end:
        time.sleep(0.001)
    return srv.poll(rid) == 1


def _finish(srv, ids):
    for rid in ids:
        srv.hold(rid, False)
    t_end = time.time() + 60
    while any(srv.poll(r) in (0, 1) for r in ids) and time.time() < t_end:
        time.sleep(0.005)
    return [srv.result(r, config=False) for r in ids]


def _alone(g, betas, seed):
    with B.Annealer.from_graph(g) as a:
        a.anneal(betas, R, 2, seed)
        return a.best_record()


@pytest.mark.parametrize("variant", [1, 3])
def test_requests_of_bit_rows_share_a_budget(variant):
    """Two populations of 4 MB, 98 MB as bytes and fields, under 64 MB."""
    require_gpu()
    g, betas = wl.gnm(*G, seed=3), wl.linear_betas(0.1, 3.0, K)
    with B.Server(64 << 20, n_streams=4, steps_per_tick=2) as srv:
        ids = []
        for seed in (1, 2):
            ids.append(srv.submit(g, betas, R, 2, seed, variant=variant))
            srv.hold(ids[-1])
            assert _running(srv, ids[-1])
        assert srv.stats()["running"] == 2
        assert srv.stats()["bytes_in_use"] <= 64 << 20
        for seed, r in zip((1, 2), _finish(srv, ids)):
            assert (r["energy"], r["step"], r["sweep"], r["slot"]) == _alone(g, betas, seed)
        assert srv.stats()["bytes_in_use"] == 0


def test_automatic_layout_is_charged_what_it_holds():
    """Admitted as the larger layout, charged as the one it got."""
    require_gpu()
    g, betas = wl.gnm(*G, seed=3), wl.linear_betas(0.1, 3.0, K)
    with B.Server(1 << 30, n_streams=4, steps_per_tick=2) as srv:
        rid = srv.submit(g, betas, R, 2, 1)
        srv.hold(rid)
        assert _running(srv, rid)
        used = srv.stats()["bytes_in_use"]
        rows = 2 * R * ((G[0] + 127) // 128 * 16)
        assert rows < used < 2 * rows + (2 << 20)
        assert _finish(srv, [rid])[0]["status"] == 0
        assert srv.stats()["bytes_in_use"] == 0
