"""The leading classes of the streamed schedule (run over all SMs through tagged loads) against the
FP64 oracle: graphs whose classes sit around the sizes where the leading part begins (64 edges)
and where its two launches meet (4,096), all of them or none in it, unit and weighted, a hub in
every class, and repeated passes (every pass starts from fresh tags)."""
import numpy as np
import pytest

import synth
from _oracle_side import assert_same_schedule
from test_gpu_parity import load_tol

pytestmark = pytest.mark.gpu

CASES = {
    "matchings_63": lambda: synth.small_family("path", 64),                       # classes below 64 edges
    "matchings_130": lambda: synth.small_family("cycle", 260),                    # classes of 64 edges and more
    "regular": lambda: synth.erdos_renyi(400, 0.9, seed=5),                       # every class large but the last
    "hubs": lambda: synth.chung_lu(20000, 200000, 2.1, seed=9, block_size=80, block_p=0.7),
    "large_classes": lambda: synth.chung_lu(60000, 240000, 2.8, seed=10),        # classes beyond 4,096 edges
}


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
@pytest.mark.parametrize("case", list(CASES))
def test_leading_classes_against_oracle(pkg, orc, case, weighted):
    import torch
    g = CASES[case]()
    w = synth.quantise_weights(np.random.default_rng(len(case)).lognormal(0, 1, g.m)) if weighted else None
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    pkg.lowd_iterate(h, 3, schedule=2)
    pkg.lowd_iterate(h, 2, schedule=2)
    info = pkg.lowd_get_info(h)
    assert info["schedule"] == 2 and info["sweep_kernel"] == 4, info
    perm, offs = (x.cpu().numpy() for x in pkg.lowd_get_edge_order(h))
    order = assert_same_schedule(orc, g.n, g.u, g.v, perm, offs, level=True)
    o = orc.LowdState(g.n, g.u, g.v, None if w is None else w.astype(np.float64))
    o.iterate(5, order=order)
    lg = pkg.lowd_get_loads(h).cpu().numpy().astype(np.float64)
    err = np.max(np.abs(lg - o.l)) / max(1.0, o.l.max())
    assert err <= load_tol(5, 4), (case, weighted, err)
    pkg.lowd_free(h)
