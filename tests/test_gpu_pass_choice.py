"""The wavefronts walk every step of a pass, the one-CTA kernels only the classes that hold edges: a graph
whose colouring is mostly empty classes, or whose classes are cheap there, keeps the one-CTA kernel that
is faster for it, and dense ones run as wavefronts.  The splits to the bit against an FP32 replay."""
import numpy as np
import pytest

from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu

# nodes, edges, kernel by its arithmetic, wavefronts
CASES = [(10001, 300, 2, False), (10002, 300, 2, False), (10001, 2500, 1, False), (10002, 2500, 1, False),
         (10001, 9000, 1, False), (10002, 9000, 1, False), (10001, 200000, 1, False), (10002, 1200000, 1, False),
         (10001, 2000000, 1, True), (1031, 250, 2, False), (1031, 20000, 1, False), (1030, 400000, 1, False),
         (1031, 250000, 1, True), (307, 60, 2, False), (307, 400, 2, True), (308, 2000, 2, True)]


def random_graph(n, m, seed):
    rng = np.random.default_rng(seed)
    key = np.zeros(0, np.int64)
    while key.size < m:
        a, b = rng.integers(0, n, 2 * m + 64), rng.integers(0, n, 2 * m + 64)
        k = np.minimum(a, b) * np.int64(n) + np.maximum(a, b)
        key = np.unique(np.concatenate([key, k[a != b]]))
    key = np.sort(rng.permutation(key)[:m])
    return (key // n).astype(np.int32), (key % n).astype(np.int32)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n,m,kernel,waves", CASES)
def test_choice_of_the_pass_kernel(n, m, kernel, waves, weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    u, v = random_graph(n, m, n + m)
    w = np.random.default_rng(m).integers(1, 9, m).astype(np.float32) if weighted else None
    h = pkg.lowd_load_graph(n, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    s0 = grid_splits(m, w, n)
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, 2, rederive_every=-1)
    info = pkg.lowd_get_info(h)
    assert info["sweep_kernel"] == kernel and (info["wavefront_blocks"] > 0) == waves, info
    got = pkg.lowd_get_splits(h).cpu().numpy()
    assert np.array_equal(got, replay(n, u, v, w, s0, 2, kernel == 1)), (n, m, weighted)
    pkg.lowd_free(h)
