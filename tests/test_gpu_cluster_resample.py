"""The one-cluster resampling kernels at the edges of their shapes (slots per
thread 1, 2, 4, 8; CTAs 1 to 8; padded ends) and the row gather at every
alignment, against the oracle and plain indexing."""
import math

import numpy as np
import pytest

import oracle
from gpu_helpers import require_gpu
from paper_2510_21105_gb300 import binding as B
from paper_2510_21105_gb300 import sharded

pytestmark = pytest.mark.gpu


def _energies(R, seed):
    rng = np.random.default_rng(seed)
    E = np.round(rng.normal(-9000.0, 150.0, R)).astype(np.int32)
    E[rng.integers(0, R)] -= 700   # a distance of ten bits: table and remaining products
    return E


@pytest.mark.parametrize("R", [2, 31, 33, 1023, 1024, 1025, 2049, 8192, 8193, 16383, 16385])
def test_noalloc_shapes(R):
    require_gpu()
    import torch

    E = _energies(R, R)
    Ed = torch.from_numpy(E).cuda()
    parent = torch.full((R,), -1, dtype=torch.int32, device="cuda")
    counts = torch.full((R,), -1, dtype=torch.int32, device="cuda")
    res = B.pa_resample_noalloc(Ed.data_ptr(), R, 1.0, 1.01, 5, 2, parent.data_ptr(), counts.data_ptr(),
                                B.current_stream_handle())
    ref = oracle.resample(E, math.exp(-(1.01 - 1.0)), sharded.resample_offset(5, 2))
    np.testing.assert_array_equal(counts.cpu().numpy(), ref["counts"])
    np.testing.assert_array_equal(parent.cpu().numpy(), ref["parent"])
    assert np.float64(res["A"]).view(np.uint64) == np.float64(ref["A"]).view(np.uint64)
    assert res["T"] == ref["T"] and res["emin"] == ref["emin"]


@pytest.mark.parametrize("R", [1, 512, 2048, 16384, 32768, 65536])
def test_shard_partials_shapes(R):
    require_gpu()
    import torch

    E = _energies(R, R + 1)
    Ed = torch.from_numpy(E).cuda()
    sh = sharded.LibraryShard(R, "cuda", stream=B.current_stream_handle())
    emin = sh.emin(Ed)
    A, T = sh.partials(Ed, emin, 1.0, 1.01)
    o = sharded.resample_offset(9, 4)
    src, counts = sh.parents(R, o, sharded.plan(1, 0, R, [A], [T], o))
    ref = oracle.resample(E, math.exp(-(1.01 - 1.0)), o)
    assert np.float64(A).view(np.uint64) == np.float64(ref["A"]).view(np.uint64) and T == ref["T"]
    np.testing.assert_array_equal(counts.cpu().numpy(), ref["counts"])
    np.testing.assert_array_equal(src.cpu().numpy(), ref["parent"])


@pytest.mark.parametrize("ncols", [1, 7, 12, 16, 19, 48, 1001, 2064, 4099])
def test_gather_alignments(ncols):
    require_gpu()
    import torch

    rng = np.random.default_rng(ncols)
    rows = 37
    src = torch.from_numpy(np.sort(rng.integers(0, rows, 50)).astype(np.int32)).cuda()
    for a, b in [(0, 0), (1, 0), (0, 3), (2, 1), (16, 32)]:
        buf = torch.from_numpy(rng.integers(-128, 128, rows * ncols + a, dtype=np.int8)).cuda()
        spins = buf[a:].view(rows, ncols)
        out = torch.full((50 * ncols + b + 8,), 99, dtype=torch.int8, device="cuda")
        rc = B.lib().pa_shard_gather(spins.data_ptr(), None, ncols, src.data_ptr(), 50, out.data_ptr() + b, None,
                                     B.current_stream_handle())
        assert rc == 0
        torch.cuda.synchronize()
        assert torch.equal(out[b:b + 50 * ncols].view(50, ncols), spins[src.long()])
        assert (out[:b] == 99).all() and (out[b + 50 * ncols:] == 99).all()
