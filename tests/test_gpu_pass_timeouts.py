"""Failure detection without a GPU fault: the waits between blocks of the wavefronts and of the level
order's leading classes give up after their limit, each with its own error bit and message, and the
context keeps working."""
import time

import numpy as np
import pytest

import synth
from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which,bit,text", [(0, 8, "wavefronts"), (1, 2, "across the grid")])
def test_waits_expire_and_report(which, bit, text):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    assert pkg.lowd_selftest_pass_timeout(2)[0] == pkg.LOWD_ERR_INVALID_ARG
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    status, bits, message = pkg.lowd_selftest_pass_timeout(which)
    assert status == pkg.LOWD_OK and bits == bit and text in message, (status, bits, message)
    assert time.perf_counter() - t0 < 10.0
    g = synth.erdos_renyi(1031, 0.5, seed=9)
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda())
    s0 = grid_splits(g.m, None, 9)
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, 2, rederive_every=-1)
    assert pkg.lowd_get_info(h)["wavefront_blocks"] > 0
    assert np.array_equal(pkg.lowd_get_splits(h).cpu().numpy(), replay(g.n, g.u, g.v, None, s0, 2, True))
    pkg.lowd_free(h)
