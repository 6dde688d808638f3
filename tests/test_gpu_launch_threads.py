"""Threads that launch the same pass kernel at the same time for graphs that need different amounts of
shared memory: the limit a kernel is given is the same for all of them, so that no thread lowers it
between another's setting and launch."""
import threading

import pytest

import synth

pytestmark = pytest.mark.gpu

GROUPS = {  # nodes, density, node versions: graphs of one kernel
    "wavefronts_one_block": [(61, 0.5, False), (131, 0.5, False), (195, 0.5, False), (259, 0.5, False)],
    "wavefronts": [(1031, 0.6, False), (2600, 0.95, False), (1031, 0.6, False), (2600, 0.95, False)],
    "staged": [(800, 0.1, False), (1030, 0.2, False), (1200, 0.1, False), (1500, 0.2, False)],
    "versions": [(300, 0.3, True), (500, 0.3, True), (800, 0.3, True), (1031, 0.3, True)],
    "ring": [(1031, 0.0005, False), (2047, 0.0001, False), (4047, 0.00003, False), (9109, 0.000005, False)],
}


@pytest.mark.parametrize("group", list(GROUPS))
def test_threads_of_one_kernel(group):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    handles = []
    for i, (n, p, versions) in enumerate(GROUPS[group]):
        g = synth.erdos_renyi(n, p, seed=i + 1)
        h = pkg.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                                stream=torch.cuda.Stream())
        pkg.lowd_iterate(h, 1, schedule=1, node_versions=versions)
        handles.append((h, versions))
    kernels = {(i["sweep_kernel"], i["wavefront_blocks"] > 0) for i in (pkg.lowd_get_info(h) for h, _ in handles)}
    assert len(kernels) == 1, kernels
    errors = []
    start = threading.Barrier(len(handles))

    def work(h, versions):
        try:
            torch.cuda.set_device(0)
            start.wait()
            for _ in range(1500):
                if errors:
                    return
                pkg.lowd_iterate(h, 1, schedule=1, node_versions=versions, rederive_every=-1)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=x) for x in handles]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for h, _ in handles:
        pkg.lowd_free(h)
