"""The exported edge order is the class-major one of the staged sweeps whichever kernel runs the passes:
the same list from wavefronts and from a handle that asked for per-node versions, before and after a
handle changes from one to the other, with and without hub stars."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,stars", [(60, 0.5, 0), (61, 0.5, 0), (330, 0.4, 0), (1031, 0.6, 0), (1031, 0.6, 600)])
def test_same_order_from_either_kernel(n, p, stars):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    g = synth.erdos_renyi(n, p, seed=n)

    def order(h):
        return [x.cpu().numpy() for x in pkg.lowd_get_edge_order(h)]

    waves = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda())
    pkg.lowd_iterate(waves, 1, hub_stars=stars)
    assert pkg.lowd_get_info(waves)["wavefront_blocks"] > 0
    other = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda())
    pkg.lowd_iterate(other, 1, hub_stars=stars, node_versions=True)
    assert pkg.lowd_get_info(other)["sweep_kernel"] == 5
    a, b = order(waves), order(other)
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
    assert np.array_equal(np.sort(a[0]), np.arange(g.m))
    if stars:
        assert 0 < pkg.lowd_get_info(waves)["star_edges"] < g.m
    pkg.lowd_iterate(waves, 1, hub_stars=stars, node_versions=True)
    assert pkg.lowd_get_info(waves)["sweep_kernel"] == 5
    assert all(np.array_equal(x, y) for x, y in zip(a, order(waves)))
    pkg.lowd_free(waves)
    pkg.lowd_free(other)
