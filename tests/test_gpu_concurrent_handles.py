"""Handles on their own streams and threads at the same time: wavefronts of several blocks that share the
GPU, a one-block handle, and a level-order handle, each to the bit what it computes alone."""
import threading

import numpy as np
import pytest

import synth
from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu


def test_handles_at_the_same_time():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    sizes = [(1031, 0.5, 0), (71, 0.5, 0), (2601, 0.3, 0), (1031, 0.4, 2), (2600, 0.95, 0), (1201, 0.5, 0)] * 2
    jobs = []
    for i, (n, p, schedule) in enumerate(sizes):
        g = synth.erdos_renyi(n, p, seed=100 + i)
        s0 = grid_splits(g.m, None, i)
        stream = torch.cuda.Stream()
        h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(), stream=stream)
        pkg.lowd_iterate(h, 0, schedule=schedule)
        jobs.append((g, s0, torch.from_numpy(s0).cuda(), schedule, h))
    torch.cuda.synchronize()

    def solve(job):
        pkg.lowd_set_splits(job[4], job[2])
        pkg.lowd_iterate(job[4], 4, rederive_every=-1, schedule=job[3])
        return pkg.lowd_get_splits(job[4]).cpu().numpy()

    alone = [solve(j) for j in jobs]
    together, errors = [None] * len(jobs), []
    start = threading.Barrier(len(jobs))

    def work(i):
        try:
            torch.cuda.set_device(0)
            start.wait()
            for _ in range(5):
                together[i] = solve(jobs[i])
        except Exception as e:
            errors.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i, (g, s0, _, schedule, h) in enumerate(jobs):
        assert np.array_equal(alone[i], together[i]), i
        info = pkg.lowd_get_info(h)
        assert (info["wavefront_blocks"] > 0) == (schedule == 0), (i, info)
        if schedule == 0:
            assert np.array_equal(alone[i], replay(g.n, g.u, g.v, None, s0, 4, info["sweep_kernel"] == 1)), i
        pkg.lowd_free(h)
