"""Child process of test_gpu_alloc_failures.py: argv[1] is a library in which the k-th allocation from the
pool can be made to fail on the host (lowd_test_fail_at)."""
import ctypes as C
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import numpy as np
import torch

import synth
from paper_2307_15969_gb300 import lowd

lib = lowd.load_library(sys.argv[1])
left = C.c_long.in_dll(lib, "lowd_test_fail_at")


def load(g, w):
    return lowd.lowd_load_graph(g.n, torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda(),
                                None if w is None else torch.from_numpy(w).cuda())


def splits(h):
    return lowd.lowd_get_splits(h).cpu().numpy()


def same(a, b):
    """Equal but for the order in which FP64 load sums are added."""
    return np.allclose(a, b, rtol=0, atol=1e-6)


def attempt(k, call):
    """The call with its k-th allocation failing: (it succeeded, an allocation did fail)."""
    left.value = k
    try:
        call()
        ok = True
    except lowd.LowdError as e:
        assert e.status == lowd.LOWD_ERR_OUT_OF_MEMORY, e
        ok = False
    failed = left.value == 0
    left.value = 0
    return ok, failed


def moving(g, w, **kw):
    """Iterate as wavefronts, then ask for node versions: whichever allocation fails, the splits are the
    ones before the call or after it, and the passes go on from there."""
    h = load(g, w)
    lowd.lowd_iterate(h, 3, **kw)
    assert lowd.lowd_get_info(h)["wavefront_blocks"] > 0
    before = splits(h)
    lowd.lowd_iterate(h, 2, node_versions=True, **kw)
    assert lowd.lowd_get_info(h)["sweep_kernel"] == 5
    after = splits(h)
    assert not same(before, after)
    lowd.lowd_free(h)
    k, stayed = 1, 0
    while True:
        h = load(g, w)
        lowd.lowd_iterate(h, 3, **kw)
        ok, failed = attempt(k, lambda: lowd.lowd_iterate(h, 2, node_versions=True, **kw))
        s = splits(h)
        assert same(s, after) or (not ok and np.array_equal(s, before)), k
        if ok and failed:
            stayed += lowd.lowd_get_info(h)["wavefront_blocks"] > 0
        if not same(s, after):
            lowd.lowd_iterate(h, 2, **kw)
            assert same(splits(h), after), k
        lowd.lowd_free(h)
        if not failed:
            break
        k += 1
    assert k > 10 and stayed > 5, (k, stayed)


def first(g, w, **kw):
    """The first iterate of a handle: whichever allocation fails, the next call starts afresh, also without
    the hub stars the failed one asked for."""
    want = []
    for opt in (kw, {}):
        h = load(g, w)
        lowd.lowd_iterate(h, 3, **opt)
        want.append((splits(h), lowd.lowd_get_info(h)))
        lowd.lowd_free(h)
    k = 1
    while True:
        h = load(g, w)
        ok, failed = attempt(k, lambda: lowd.lowd_iterate(h, 3, **kw))
        info = lowd.lowd_get_info(h)
        if ok:
            assert same(splits(h), want[0][0]), k
        elif info["classes"] == 0:   # nothing was prepared
            assert info["star_steps"] == 0 and info["star_edges"] == 0, k
            lowd.lowd_iterate(h, 3)
            assert same(splits(h), want[1][0]), k
            assert lowd.lowd_get_info(h)["star_edges"] == want[1][1]["star_edges"]
        lowd.lowd_free(h)
        if not failed:
            break
        k += 1
    assert k > 10, k


def main():
    g = synth.erdos_renyi(1031, 0.6, seed=3)
    w = np.random.default_rng(3).integers(1, 9, g.m).astype(np.float32)
    c = synth.chung_lu(1031, 200000, 2.1, seed=5, block_size=400, block_p=0.9)
    moving(g, None)
    moving(g, w)
    moving(c, None, hub_stars=1)
    first(g, w)
    first(c, None, hub_stars=1)
    first(c, None, schedule=2)
    print("ALLOC_OK")


main()
