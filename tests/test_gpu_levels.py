"""The level colouring's frontiers on one SM, where they fit its shared memory (4,096 ranks) and
where they grow beyond it again: a tree whose degrees grow with the depth starts with a single
ready edge and fans out over a regular last layer.  The schedule must be the oracle's own."""
import numpy as np
import pytest

from _oracle_side import assert_same_schedule

pytestmark = pytest.mark.gpu


def fan_out(depth, regular):
    """Nodes at depth d have d + 1 children (two at the root and below it); the last layer is
    joined in a circulant of `regular` neighbours, so that its degree is the largest."""
    u, v, layer, nxt = [], [], np.array([0]), 1
    for d in range(depth):
        c = max(2, d + 1)
        kids = np.arange(nxt, nxt + c * layer.size)
        u.append(np.repeat(layer, c))
        v.append(kids)
        layer, nxt = kids, nxt + kids.size
    k = layer.size
    for s in range(1, regular // 2 + 1):
        u.append(layer)
        v.append(np.roll(layer, -s))
    if regular % 2:
        u.append(layer[:k // 2])
        v.append(layer[k // 2:])
    u, v = np.concatenate(u), np.concatenate(v)
    return nxt, np.minimum(u, v).astype(np.int32), np.maximum(u, v).astype(np.int32)


@pytest.mark.parametrize("depth,regular,beyond", [(5, 7, False), (7, 8, False), (8, 9, True)])
def test_frontiers_on_one_sm(depth, regular, beyond):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2307_15969_gb300 import build
    build.build()
    oracle.build()
    import paper_2307_15969_gb300 as pkg
    n, u, v = fan_out(depth, regular)
    order = np.lexsort((v, u))
    u, v = u[order], v[order]
    h = pkg.lowd_load_graph(n, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda())
    pkg.lowd_iterate(h, 1, schedule=2)
    perm, offs = (x.cpu().numpy() for x in pkg.lowd_get_edge_order(h))
    sizes = np.diff(offs)
    assert sizes[0] < 4096 and (sizes.max() > 4096) == beyond, (sizes[0], sizes.max())
    assert_same_schedule(oracle, n, u, v, perm, offs, level=True)
    pkg.lowd_free(h)
