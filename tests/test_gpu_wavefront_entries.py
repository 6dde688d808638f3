"""The last inputs of a lap: a tile of the wavefronts whose inputs run out inside a group of four steps.

The last high tile holds one row at n = 64 k + 3 (and 64 k + 4 with the odd node), so the entries that
end a lap come from the warps of two tiles, in no order of their own; each is used only once its tag is
seen.  The splits after several passes in one launch are those of an FP32 replay, to the bit, on one block
and on several, with and without the odd node, with single FP32 and with pair loads, again and again.
"""
import numpy as np
import pytest

import synth
from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n,p", [(67, 0.7), (68, 0.7), (131, 0.5), (132, 0.5), (195, 0.4), (196, 0.4), (259, 0.4),
                                 (260, 0.4), (323, 0.4), (324, 0.4), (515, 0.3), (708, 0.97), (1027, 0.3)])
def test_last_entries_of_a_lap(n, p, weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    g = synth.erdos_renyi(n, p, seed=n)
    w = synth.quantise_weights(np.random.default_rng(n).lognormal(0, 1, g.m)) if weighted else None
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    s0 = grid_splits(g.m, w, n + 1)
    want = None
    for _ in range(4):
        pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
        pkg.lowd_iterate(h, 6, rederive_every=-1)
        if want is None:
            want = replay(g.n, g.u, g.v, w, s0, 6, pkg.lowd_get_info(h)["sweep_kernel"] == 1)
        got = pkg.lowd_get_splits(h).cpu().numpy()
        assert np.array_equal(got, want), (n, weighted, int((got != want).sum()))
    pkg.lowd_free(h)
