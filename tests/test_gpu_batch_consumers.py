"""The batched passes with as many consumer threads as the longest class has edges, and with fewer
(several edges per thread): complete graphs whose classes hold 31 to 33 edges and 128 or 129,
against the oracle's passes."""
import numpy as np
import pytest

from _oracle_side import oracle_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [64, 96, 256, 512])
def test_consumers_per_class(threads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import synth
    from paper_2307_15969_gb300 import build
    build.build()
    oracle.build()
    import paper_2307_15969_gb300 as pkg
    graphs = []
    for n in (63, 64, 66, 67, 257, 258, 259):
        u, v = np.triu_indices(n, 1)
        keep = (u * 7 + v) % 97 != 0          # some classes lose edges, the loads differ
        graphs.append(synth.Graph(n, u[keep].astype(np.int32), v[keep].astype(np.int32), None))
    node_off = np.concatenate([[0], np.cumsum([g.n for g in graphs])]).astype(np.int64)
    edge_off = np.concatenate([[0], np.cumsum([g.m for g in graphs])]).astype(np.int64)
    b = pkg.lowd_batch_create(node_off, edge_off, np.concatenate([g.u for g in graphs]),
                              np.concatenate([g.v for g in graphs]))
    T = 7
    pkg.lowd_batch_run(b, passes=T, threads=threads)
    loads, status = pkg.lowd_batch_loads(b), pkg.lowd_batch_results(b)["status"]
    for i, g in enumerate(graphs):
        assert status[i] == 0
        nh, uh, vh, _, idmap = oracle_graph(oracle, g, True)
        order, _, _ = oracle.circle_order(nh, uh, vh)
        o = oracle.LowdState(nh, uh, vh)
        o.iterate(T, order=order)
        err = np.max(np.abs(loads[node_off[i]:node_off[i + 1]].astype(np.float64)[idmap] - o.l))
        assert err <= 1e-4 * max(1.0, o.l.max()), (g.n, threads, err)   # single FP32 loads
    pkg.lowd_batch_free(b)
