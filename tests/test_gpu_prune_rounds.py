"""Algorithm 2's rounds in one launch, bit for bit against the oracle: no round at all, one round,
many rounds (a clique with ever sparser shells around it), sizes around a tile of 2,048 edges and
its multiples, several blocks, unit and weighted."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _shells(layers):
    """A 12-clique, then layers of nodes hanging on the layer before by ever fewer edges."""
    pairs = [(i, j) for i in range(12) for j in range(i + 1, 12)]
    prev, n = list(range(12)), 12
    for k in range(layers):
        cur = list(range(n, n + 12 + 4 * k))
        pairs += [(prev[(i + t) % len(prev)], x) for i, x in enumerate(cur) for t in range(max(1, 5 - k // 2))]
        prev, n = cur, n + len(cur)
    return synth.graphs._from_pairs(n, pairs)


CASES = {
    "no_edges": lambda: synth.small_family("empty", 40),
    "no_round": lambda: synth.small_family("clique", 9),
    "one_round": lambda: synth.small_family("star", 300),
    "shells": lambda: _shells(14),
    "tile_below": lambda: synth.planted_background(1000, 3.7, 40, 0.3, seed=3),
    "tile_above": lambda: synth.planted_background(1100, 4.0, 60, 0.4, seed=4),
    "blocks": lambda: synth.chung_lu(9000, 70000, 2.2, seed=5, block_size=50, block_p=0.6),
    "many_blocks": lambda: synth.rmat(16, 16, 0.57, 0.19, 0.19, seed=6, block_size=128, block_p=0.5),
}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_prune_rounds_bit_exact(case, weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import oracle
    import paper_2307_15969_gb300 as pkg
    oracle.build()
    g = CASES[case]()
    w = None
    if weighted:
        w = synth.quantise_weights(np.random.default_rng(7).lognormal(0, 1, g.m)) if g.m else np.zeros(0, np.float32)
    h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    nk, mk, rounds = pkg.lowd_prune(h)
    _, rr = (x.cpu().numpy() for x in pkg.lowd_get_prune_info(h))
    wu, _ = oracle.weight_units(g.m, None if w is None else w.astype(np.float64))
    pr = oracle.prune(g.n, g.u, g.v, wu, weighted)
    want = np.asarray(pr["removal_round"])
    assert np.array_equal(rr, want), case
    assert rounds == max(int(want.max(initial=-1)), 0)
    keep = want < 0
    assert nk == int(keep.sum()) and mk == int((keep[g.u] & keep[g.v]).sum())
    u, v, _ = (x.cpu().numpy() for x in pkg.lowd_get_graph(h))
    new = np.cumsum(keep) - 1
    ke = keep[g.u] & keep[g.v]
    assert np.array_equal(u, new[g.u[ke]]) and np.array_equal(v, new[g.v[ke]])
    pkg.lowd_free(h)
