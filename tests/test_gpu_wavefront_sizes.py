"""Wavefronts at sizes above those of one or two pairs of tiles per SM, to the bit against an FP32 replay:
an even node count with many tiles (its low tiles wait input by input at a lap's end), four pairs of tiles
per block for an odd one, and single FP32 loads where pairs would not fit the staged sweep."""
import numpy as np
import pytest

from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu

# nodes, density, kernel by its arithmetic, blocks
CASES = [(9110, 0.15, 1, 36), (19521, 0.066, 1, 77), (19522, 0.066, 1, 77), (26001, 0.064, 2, 102)]


def rows_graph(n, p, seed):
    """G(n, p), row by row, in canonical order."""
    rng = np.random.default_rng(seed)
    v = [a + 1 + np.flatnonzero(rng.random(n - 1 - a, dtype=np.float32) < p) for a in range(n)]
    u = np.repeat(np.arange(n), [x.size for x in v])
    return u.astype(np.int32), np.concatenate(v).astype(np.int32)


@pytest.mark.parametrize("n,p,kernel,blocks", CASES)
def test_many_tiles(n, p, kernel, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    u, v = rows_graph(n, p, n)
    passes = 2 if n < 20000 else 1
    h = pkg.lowd_load_graph(n, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda())
    s0 = grid_splits(u.size, None, n)
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, passes, rederive_every=-1)
    info = pkg.lowd_get_info(h)
    assert info["sweep_kernel"] == kernel and info["wavefront_blocks"] == blocks, info
    got = pkg.lowd_get_splits(h).cpu().numpy()
    assert np.array_equal(got, replay(n, u, v, None, s0, passes, kernel == 1))
    pkg.lowd_free(h)
