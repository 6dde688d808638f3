"""Which kernel runs a pass, by lowd_info: the wavefronts with the blocks expected of them, or the staged
sweep and its edges per thread on graphs that keep it; the splits to the bit against an FP32 replay."""
import numpy as np
import pytest

import synth
from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu

# nodes, density, versions asked for, expected kernel, edges per thread, blocks of the wavefronts
CASES = {
    "one_block": (60, 0.5, False, 2, None, lambda w: 1),
    "one_block_most": (319, 0.4, False, 2, None, lambda w: 3 if w else 1),
    "two_pairs_a_block": (1031, 0.6, False, 1, 1, lambda w: 9),
    "four_pairs_a_block": (2600, 0.95, False, 1, 2, lambda w: 11),
    "staged_e2": (2600, 0.95, True, 1, 2, lambda w: 0),
    "versions": (1031, 0.6, True, 5, 1, lambda w: 0),
}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_kernel_that_ran(case, weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    n, p, versions, kernel, edges, blocks = CASES[case]
    g = synth.erdos_renyi(n, p, seed=n)
    w = synth.quantise_weights(np.random.default_rng(n).lognormal(0, 1, g.m)) if weighted else None
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    assert pkg.lowd_get_info(h)["wavefront_blocks"] == 0
    pkg.lowd_iterate(h, 0, node_versions=versions)
    s0 = grid_splits(g.m, w, n)
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, 2, rederive_every=-1, node_versions=versions)
    info = pkg.lowd_get_info(h)
    assert info["sweep_kernel"] == kernel and info["wavefront_blocks"] == blocks(weighted), info
    if edges is not None:
        assert info["sweep_edges_per_thread"] == edges, info
    got = pkg.lowd_get_splits(h).cpu().numpy()
    assert np.array_equal(got, replay(g.n, g.u, g.v, w, s0, 2, kernel != 2)), (case, weighted)
    pkg.lowd_free(h)
