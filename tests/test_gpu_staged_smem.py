"""Staged sweeps whose stages would fill a block's shared memory to the last bytes.

227 KB hold the dynamic part and the kernel's static word (128 bytes before the aligned dynamic part).
The graphs here have the same number of edges in every colour class, so that the layout of their
largest chunk and stage count comes to exactly 227 KB (FULL: one stage fewer has to be taken) or to
227 KB less 128 bytes (FITS: it runs as it is); without and with per-node versions.  The splits are
those of an FP32 replay, to the bit.
"""
import numpy as np
import pytest

from _replay import grid_splits, replay

pytestmark = pytest.mark.gpu

CASES = [  # n, edges a class, weighted, versions
    (574, 148, False, False),   # FULL: 16 classes a chunk, 12 stages
    (760, 196, False, False),   # FULL: 9 stages
    (558, 148, False, False),   # FITS
    (1598, 76, True, False),    # FULL: 15 stages, weighted
    (558, 148, True, False),    # FITS, weighted
    (312, 108, False, True),    # FITS
    (374, 148, True, True),     # FITS, weighted
]


def _round_up(x):
    return (x + 127) & ~127


def _staged_bytes(n, C, stages, longest, weighted, per_chunk, versions):
    """Bytes of the staged layout: barriers, loads as pairs (and versions), chunk offsets, stages of
    ends, splits (, ranks) (, weights)."""
    head = 256 + 8 * (n + 1)
    if versions:
        head = (head + 4 * (n + 1) + 15) & ~15
    head += 4 * ((C + per_chunk - 1) // per_chunk + 1)
    return _round_up(head) + _round_up(4 * longest) * (2 + weighted + versions) * stages


def uniform_classes(n, k):
    """n nodes with exactly k edges in each of the circle method's classes."""
    P = n + (n & 1) - 1
    a = np.arange(P)
    us, vs = [], []
    for c in range(P):
        b = (c - a) % P
        keep = np.flatnonzero(a < b)[:k]
        assert keep.size == k
        us.append(keep)
        vs.append(b[keep])
    u, v = np.concatenate(us), np.concatenate(vs)
    order = np.lexsort((v, u))
    return u[order].astype(np.int32), v[order].astype(np.int32)


def test_the_sizes_fill_shared_memory():
    most = 227 * 1024
    for n, k, weighted, versions in CASES:
        C = n + (n & 1) - 1
        sizes = [_staged_bytes(n, C, s, 16 * ((k + 3) & ~3), weighted, 16, versions) for s in range(3, 17)]
        assert most in sizes or most - 128 in sizes, (n, k)
        assert max(x for x in sizes if x <= most) in (most, most - 128), (n, k)


@pytest.mark.parametrize("n,k,weighted,versions", CASES)
def test_full_shared_memory(n, k, weighted, versions):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    import paper_2307_15969_gb300 as pkg
    u, v = uniform_classes(n, k)
    w = np.random.default_rng(n).integers(1, 9, u.size).astype(np.float32) if weighted else None
    h = pkg.lowd_load_graph(n, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(),
                            None if w is None else torch.from_numpy(w).cuda())
    s0 = grid_splits(u.size, w, n)
    pkg.lowd_iterate(h, 0, node_versions=versions)   # the schedule as the sweep asked for reads it
    pkg.lowd_set_splits(h, torch.from_numpy(s0).cuda())
    pkg.lowd_iterate(h, 3, rederive_every=-1, node_versions=versions)
    info = pkg.lowd_get_info(h)
    assert info["classes"] == n + (n & 1) - 1 and info["sweep_kernel"] == (5 if versions else 1), info
    got = pkg.lowd_get_splits(h).cpu().numpy()
    assert np.array_equal(got, replay(n, u, v, w, s0, 3, True))
    pkg.lowd_free(h)
