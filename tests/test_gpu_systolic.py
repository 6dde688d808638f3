"""The systolic passes against the FP64 oracle at the edges of their tiles.

A pass runs the circle colouring's classes as wavefronts over tiles of 32 rows, two tiles per
warp, several warps per block, and streams between blocks; an even node count adds the odd
node of the colouring, whose load travels along the diagonal.  The sizes sit on both sides of
one tile, two tiles, one block (512 nodes) and several blocks, and of the switch from single
FP32 to pair loads.  Loads are held to the bar of the arithmetic that ran (1e-6 of the largest
load for pairs, 1e-4 for single FP32); two calls, so that a cut at a pass boundary is resumed.
"""
import numpy as np
import pytest

import synth
from _oracle_side import assert_same_schedule
from test_gpu_parity import load_tol

pytestmark = pytest.mark.gpu

SIZES = [9, 10, 31, 33, 34, 63, 64, 65, 66, 67, 68, 69, 71, 72, 73, 128, 129, 130, 255, 384, 385, 386, 511, 512, 513, 514, 577, 770, 1030, 1090]


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as p
    p.load_library()
    return p


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_systolic_pass_against_oracle(pkg, orc, n, weighted):
    import torch
    # even sizes above 384 run on the array only with at least 320 edges a class
    g = synth.erdos_renyi(n, 0.9 if n < 40 else (0.95 if n >= 700 else 0.3), seed=n)
    w = synth.quantise_weights(np.random.default_rng(n).lognormal(0, 1, g.m)) if weighted else None
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    s0 = np.random.default_rng(n + 1).random(g.m).astype(np.float32)   # uneven start: transfers clip at both ends
    if w is not None:
        s0 = (s0 * w).astype(np.float32)
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, 2)
    pkg.lowd_iterate(h, 3)
    info = pkg.lowd_get_info(h)
    assert info["sweep_kernel"] == (1 if n >= 384 else 2), info
    perm, offs = (x.cpu().numpy() for x in pkg.lowd_get_edge_order(h))
    order = assert_same_schedule(orc, g.n, g.u, g.v, perm, offs)
    o = orc.LowdState(g.n, g.u, g.v, None if w is None else w.astype(np.float64))
    o.fu = s0.astype(np.float64)
    o.fv = o.w - o.fu
    o.l = np.bincount(g.u, weights=o.fu, minlength=n) + np.bincount(g.v, weights=o.fv, minlength=n)
    o.iterate(5, order=order)
    lg = pkg.lowd_get_loads(h).cpu().numpy().astype(np.float64)
    err = np.max(np.abs(lg - o.l)) / max(1.0, o.l.max())
    assert err <= load_tol(5, info["sweep_kernel"]), (n, weighted, err)
    s = pkg.lowd_get_splits(h).cpu().numpy().astype(np.float64)
    wt = np.ones(g.m) if w is None else w.astype(np.float64)
    assert np.all(s >= 0) and np.all(s <= wt)
    pkg.lowd_free(h)
