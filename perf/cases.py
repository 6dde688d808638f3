"""The work a user of this package has it do, as measurable cases.

Each case is one whole use of the public entry points on a seeded synthetic graph: solve a
graph (load, prune, passes, extraction), prune it, run to a certified gap with hub stars, run
the passes on an unpruned graph, start from the learned warm start, solve a batch of graphs, or
take one training step of the warm-start network.  The graph recipes are those of the
repository's workloads (Chung-Lu with a planted block, R-MAT (.57, .19, .19, .05) with a
planted block, lognormal weights on the 2^-20 grid, the batched Chung-Lu mix), drawn on the GPU
from the seed.  ``exact`` gives what a case returns in 64-bit arithmetic, written from the
definitions of the method (Algorithms 1 and 2, the circle colouring and the level order that
fix the order of a pass, the extraction, the network).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2307_15969_gb300 as lowd
from paper_2307_15969_gb300 import warmstart

GRID = 1 << 20            # weights are multiples of 1 / GRID
EXACT_STEPS = 260_000     # class updates the 64-bit replay does in well under 20 seconds
EXACT_LEVEL_EDGES = 1_300_000

LISTED = [
    # The smallest call: a small network solved on its own, device arrays; latency and launches.
    dict(name="solve_small", kind="solve", model="chunglu", n=2000, m=8000, gamma=2.1, block=24, block_p=0.6,
         weighted=False, raw=False, host=False, prune=True, passes=200, check_every=0),
    # A citation-size network from host arrays, with the stop test evaluated along the way.
    dict(name="solve_chunglu_10k", kind="solve", model="chunglu", n=10000, m=100000, gamma=2.1, block=64,
         block_p=0.6, weighted=False, raw=False, host=True, prune=True, passes=200, check_every=50),
    # A mid-size network as it comes from an edge dump: both directions, repeats, any order.
    dict(name="solve_rmat18_raw", kind="solve", model="rmat", scale=18, ef=16, block=256, block_p=0.5,
         weighted=False, raw=True, host=False, prune=True, passes=50, check_every=0),
    # The flagship: a social-network-size graph, 200 passes on its pruned core.
    dict(name="solve_rmat22", kind="solve", model="rmat", scale=22, ef=16, block=256, block_p=0.5,
         weighted=False, raw=False, host=False, prune=True, passes=200, check_every=0),
    # A weighted graph end to end from pinned host memory.
    dict(name="solve_rmat20w_host", kind="solve", model="rmat", scale=20, ef=10, block=512, block_p=0.5,
         weighted=True, raw=False, host=True, prune=True, passes=100, check_every=0),
    # Pruning as a preprocessing service: the core, the degree order and the removal rounds.
    dict(name="prune_rmat22", kind="prune", model="rmat", scale=22, ef=16, block=256, block_p=0.5,
         weighted=False, raw=False, host=False),
    # Densest subgraph with a certificate: hub-star passes until the gap is 1e-6, then the shells.
    dict(name="certify_rmat20", kind="certify", model="rmat", scale=20, ef=16, block=256, block_p=0.5,
         weighted=False, raw=False, host=False, passes=400, check_every=10, rel_tol=1e-6),
    # The whole decomposition is wanted, so nothing is pruned: plain passes over every edge.
    dict(name="unpruned_rmat16", kind="unpruned", model="rmat", scale=16, ef=16, block=128, block_p=0.5,
         weighted=False, raw=False, host=False, passes=10, hub_stars=0),
    # The same on a larger weighted graph with hub-star updates.
    dict(name="unpruned_rmat20w_stars", kind="unpruned", model="rmat", scale=20, ef=8, block=512, block_p=0.5,
         weighted=True, raw=False, host=False, passes=5, hub_stars=1),
    # The learned warm start on a pruned core, a checkpoint of the splits, a few passes.
    dict(name="warm_rmat18", kind="warm", model="rmat", scale=18, ef=16, block=256, block_p=0.5,
         weighted=False, raw=False, host=False, passes=10),
    # Many independent small graphs through the whole method at once.
    dict(name="batch_256", kind="batch", graphs=256, n_lo=100, n_hi=20000, passes=100),
    # One training step of the warm-start network on a minibatch of 32 cores.
    dict(name="train_32", kind="train", cores=32, n_lo=60, n_hi=1200),
]


def listed():
    return [dict(c) for c in LISTED]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "prune", "certify", "unpruned", "warm", "batch", "train"])
    if kind == "batch":
        return dict(kind="batch", graphs=_log_int(rng, 1, 300), n_lo=100, n_hi=_log_int(rng, 400, 20000),
                    passes=_log_int(rng, 5, 100))
    if kind == "train":
        return dict(kind="train", cores=_log_int(rng, 1, 40), n_lo=_log_int(rng, 10, 80), n_hi=_log_int(rng, 100, 1200))
    if rng.random() < 0.5 and kind != "unpruned":
        n = _log_int(rng, 200, 60000)
        m = int(n * rng.uniform(4.0, 16.0))
        c = dict(kind=kind, model="chunglu", n=n, m=m, gamma=rng.uniform(2.1, 2.8),
                 block=max(8, _log_int(rng, 12, 400)), block_p=rng.uniform(0.4, 0.7))
    else:
        scale = rng.randint(16, 20) if kind == "unpruned" else rng.randint(12, 21)
        c = dict(kind=kind, model="rmat", scale=scale, ef=rng.randint(6, 16), block=_log_int(rng, 64, 512), block_p=0.5)
    c.update(weighted=rng.random() < 0.4, raw=rng.random() < 0.3, host=rng.random() < 0.3)
    if kind == "solve":
        c.update(prune=c["model"] == "rmat" or c["n"] > 20000 or rng.random() < 0.7, passes=_log_int(rng, 10, 200),
                 check_every=rng.choice([0, 0, 10, 50]))
        if not c["prune"]:
            c["passes"] = min(c["passes"], 30)
    elif kind == "certify":
        c.update(passes=200, check_every=10, rel_tol=rng.choice([1e-5, 1e-6]))
    elif kind == "unpruned":
        c.update(passes=rng.randint(1, 6), hub_stars=rng.choice([0, 1]))
    elif kind == "warm":
        c.update(passes=_log_int(rng, 1, 20))
    return c


# ------------------------------------------------------------------ inputs (drawn on the GPU)

def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + 7919 * stream + 12345) % (1 << 62))
    return g


def _block_keys(g, n, size, p):
    size = min(size, n)
    nodes = torch.randperm(n, generator=g, device="cuda")[:size]
    ij = torch.triu_indices(size, size, 1, device="cuda")
    keep = torch.rand(ij.shape[1], generator=g, device="cuda") < p
    a, b = nodes[ij[0][keep]], nodes[ij[1][keep]]
    return torch.minimum(a, b) * n + torch.maximum(a, b)


def _graph_keys(case, seed, stream=0):
    """(n, sorted unique keys lo * n + hi) of the case's graph."""
    g = _gen(seed, stream)
    if case["model"] == "rmat":
        scale = case["scale"]
        n = 1 << scale
        m = case["ef"] * n
        perm = torch.randperm(n, generator=g, device="cuda")
        parts = []
        for lo in range(0, m, 1 << 24):
            cnt = min(1 << 24, m - lo)
            a = torch.zeros(cnt, dtype=torch.int64, device="cuda")
            b = torch.zeros_like(a)
            for lvl in range(scale):
                r = torch.rand(cnt, generator=g, device="cuda")
                a |= (r >= 0.76).long() << lvl
                b |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << lvl
            a, b = perm[a], perm[b]
            ok = a != b
            parts.append((torch.minimum(a, b) * n + torch.maximum(a, b))[ok])
        keys = torch.cat(parts)
    else:
        n, m = case["n"], case["m"]
        wt = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (case["gamma"] - 1.0))
        p = torch.empty_like(wt)
        p[torch.randperm(n, generator=g, device="cuda")] = wt
        cdf = torch.cumsum(p, 0) / p.sum()
        a, b = (torch.searchsorted(cdf, torch.rand(m, generator=g, device="cuda", dtype=torch.float64), right=True)
                .clamp_(max=n - 1) for _ in range(2))
        ok = a != b
        keys = (torch.minimum(a, b) * n + torch.maximum(a, b))[ok]
    if case["block"] > 1:
        keys = torch.cat([keys, _block_keys(g, n, case["block"], case["block_p"])])
    return n, torch.unique(keys)


def _graph(case, seed):
    """(n, u, v, w or None): the canonical edge list and, for ``raw``, the list a user hands in."""
    n, keys = _graph_keys(case, seed)
    u, v = (keys // n).int(), (keys % n).int()
    w = None
    g = _gen(seed, 1)
    if case["weighted"]:
        x = torch.randn(u.shape[0], generator=g, device="cuda", dtype=torch.float64).exp_()
        w = (torch.round(x * GRID).clamp_(min=1.0) / GRID).float()
    raw = (u, v, w)
    if case["raw"]:
        m = u.shape[0]
        idx = torch.cat([torch.arange(m, device="cuda"), torch.randint(0, m, (m // 3,), generator=g, device="cuda")])
        idx = idx[torch.randperm(idx.shape[0], generator=g, device="cuda")]
        flip = torch.rand(idx.shape[0], generator=g, device="cuda") < 0.5
        ru, rv = torch.where(flip, v[idx], u[idx]), torch.where(flip, u[idx], v[idx])
        raw = (ru.contiguous(), rv.contiguous(), w[idx].contiguous() if w is not None else None)
    return n, (u, v, w), raw


def _pinned(t):
    if t is None:
        return None
    p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    p.copy_(t)
    return p.numpy()


def _batch_graphs(case, seed):
    """[(n, u, v)] in the batched workload's mix: n uniform, average degree 4 to 32, a 5 % block."""
    sizes = np.random.default_rng([case["graphs"], case["n_lo"], case["n_hi"]])   # the sizes are the case's
    rng = np.random.default_rng([seed, 77])
    out = []
    for i in range(case["graphs"]):
        n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
        d = float(sizes.uniform(4.0, 32.0))
        sub = dict(model="chunglu", n=n, m=min(int(round(n * d / 2)), n * (n - 1) // 4),
                   gamma=float(rng.uniform(2.1, 2.8)), block=max(2, int(round(0.05 * n))), block_p=0.5)
        _, keys = _graph_keys(sub, seed, stream=100 + i)
        out.append((n, (keys // n).int().cpu().numpy(), (keys % n).int().cpu().numpy()))
    return out


def _train_batch(case, seed):
    """A minibatch: the disjoint union of dense cores with their target loads (a core that is its
    own densest subgraph ends with every load at its density), and starting parameters."""
    sizes = np.random.default_rng([case["cores"], case["n_lo"], case["n_hi"]])   # the sizes are the case's
    rng = np.random.default_rng([seed, 78])
    lo, hi, t, off = [], [], [], 0
    for _ in range(case["cores"]):
        n = int(round(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        a = rng.uniform(0.4, 1.0, n)   # uneven degrees, as a core's
        iu, ju = np.triu_indices(n, k=1)
        keep = rng.random(iu.shape[0]) < a[iu] * a[ju]
        lo.append(iu[keep] + off)
        hi.append(ju[keep] + off)
        t.append(np.full(n, keep.sum() / n, np.float32))
        off += n
    lo, hi, t = np.concatenate(lo).astype(np.int32), np.concatenate(hi).astype(np.int32), np.concatenate(t)
    # He-uniform layers, no biases, a small readout: where training starts
    parts = [rng.uniform(-1, 1, 192) * math.sqrt(2.0), np.zeros(64)]
    for _ in range(3):
        parts += [rng.uniform(-1, 1, 8192) * math.sqrt(6.0 / 128), np.zeros(64)]
    parts.append(rng.uniform(-1, 1, 64) * 0.01)
    return off, lo, hi, t, np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        gs = _batch_graphs(case, seed)
        no = np.concatenate([[0], np.cumsum([g[0] for g in gs])]).astype(np.int64)
        eo = np.concatenate([[0], np.cumsum([g[1].shape[0] for g in gs])]).astype(np.int64)
        b = lowd.lowd_batch_create(no, eo, np.concatenate([g[1] for g in gs]), np.concatenate([g[2] for g in gs]))
        return dict(kind=kind, case=case, batch=b)
    if kind == "train":
        n, lo, hi, t, params = _train_batch(case, seed)
        return dict(kind=kind, case=case, net=lowd.lowd_mpnn_create(), n=n, lo=lo, hi=hi, t=t, params=params)
    n, _, (u, v, w) = _graph(case, seed)
    if case["host"]:
        u, v, w = _pinned(u), _pinned(v), _pinned(w)
    st = dict(kind=kind, case=case, n=n, u=u, v=v, w=w)
    if kind == "warm":
        st["net"] = lowd.lowd_mpnn_create()
        lowd.lowd_mpnn_set_params(st["net"], warmstart.load_params())
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass

def _members(S, n):
    """S as one byte per node: 1 for its members."""
    if isinstance(S, np.ndarray):
        x = np.zeros(n, np.uint8)
        x[S] = 1
        return x
    return torch.zeros(n, dtype=torch.uint8, device=S.device).index_fill_(0, S.long(), 1)


def _at_shell(lam, shell):
    """Each node's shell density; 0 for pruned nodes (shell 0)."""
    if isinstance(lam, np.ndarray):
        return np.concatenate([[0.0], lam])[shell]
    return torch.cat([lam.new_zeros(1), lam])[shell.long()]


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "batch":
        b = state["batch"]
        lowd.lowd_batch_run(b, passes=case["passes"])
        out = lowd.lowd_batch_results(b)
        out["loads"] = lowd.lowd_batch_loads(b)
        return out
    if kind == "train":
        net = state["net"]
        lowd.lowd_mpnn_set_params(net, state["params"])
        lowd.lowd_mpnn_bind(net, state["n"], state["lo"], state["hi"], None, state["t"])
        loss = lowd.lowd_mpnn_forward(net)
        loads = lowd.lowd_mpnn_read(net, lowd.LOWD_MPNN_LOADS)
        lowd.lowd_mpnn_backward(net)
        lowd.lowd_mpnn_adam(net, 1e-3)
        return dict(loss=loss, loads=loads, grad=lowd.lowd_mpnn_read(net, lowd.LOWD_MPNN_GRAD),
                    params=lowd.lowd_mpnn_get_params(net))
    h = lowd.lowd_load_graph(state["n"], state["u"], state["v"], state["w"])
    out = {}
    if kind in ("prune", "certify", "warm") or case.get("prune"):
        out["kept"], out["kept_edges"], out["rounds"] = lowd.lowd_prune(h)
    if kind == "prune":
        out["order"], out["removal_round"] = lowd.lowd_get_prune_info(h)
    elif kind == "solve":
        st = lowd.lowd_iterate(h, case["passes"], check_every=case["check_every"])
        out.update(sum_load_sq=st["sum_load_sq"], max_load=st["max_load"])
    elif kind == "certify":
        st = lowd.lowd_iterate(h, case["passes"], check_every=case["check_every"], rel_tol=case["rel_tol"], hub_stars=1)
        out.update(passes=st["iters_done"], converged=st["converged"], max_load=st["max_load"])
        out["shell"], lam, _ = lowd.lowd_get_ldd(h, rel_tol=1e-3)
        out["shell_density"] = _at_shell(lam, out["shell"])
    elif kind == "unpruned":
        st = lowd.lowd_iterate(h, case["passes"], hub_stars=case["hub_stars"])
        out.update(sum_load_sq=st["sum_load_sq"], max_load=st["max_load"])
    elif kind == "warm":
        lowd.lowd_warm_start(h, state["net"])
        out["start_loads"] = lowd.lowd_extract(h)[2]
        st = lowd.lowd_iterate(h, case["passes"])
        out.update(sum_load_sq=st["sum_load_sq"], max_load=st["max_load"])
    S, out["rho"], out["loads"] = lowd.lowd_extract(h)
    out["S"] = _members(S, state["n"])
    lowd.lowd_free(h)
    return out


# ------------------------------------------------------------------ what a pass cannot do without

def _core_edges(case):
    """Rough size of the pruned core: the passes' edges (R-MAT cores grow slower than the graph)."""
    if case["model"] == "rmat":
        m = case["ef"] << case["scale"]
        return min(m, 0.1 * m * 2.0 ** (0.33 * (22 - case["scale"])) * case["ef"] / 16.0)
    return 0.3 * case["m"] + case["block"] ** 2 * case["block_p"] / 2


def work(case):
    """Every input read once, every output written once; 8 flops per edge update of a pass (the
    difference, its half, the two clips, the two load changes and the split)."""
    kind = case["kind"]
    if kind == "batch":
        nodes = case["graphs"] * (case["n_lo"] + case["n_hi"]) / 2
        edges = nodes * 9.0 + case["graphs"] * 0.25 * (0.05 * (case["n_lo"] + case["n_hi"]) / 2) ** 2
        return dict(bytes=int(8 * edges + 5 * nodes), flops=int(8 * 0.5 * edges * case["passes"]))
    if kind == "train":
        n1 = (case["n_hi"] - case["n_lo"]) / max(math.log(case["n_hi"] / case["n_lo"]), 1e-9)
        n2 = (case["n_hi"] ** 2 - case["n_lo"] ** 2) / (2 * max(math.log(case["n_hi"] / case["n_lo"]), 1e-9))
        n, m = case["cores"] * n1, case["cores"] * n2 / 4
        return dict(bytes=int(8 * m + 8 * n + 4 * 25088 * 3), flops=int(n * 3 * 3 * 2 * 128 * 64 + m * 64 * 2 * 2 * 6))
    m = (case["ef"] << case["scale"]) if case["model"] == "rmat" else case["m"]
    n = (1 << case["scale"]) if case["model"] == "rmat" else case["n"]
    m += case["block"] ** 2 * case["block_p"] / 2
    per = 12 if case["weighted"] else 8
    b = m * per * (4 / 3 if case["raw"] else 1) + 8 * n
    if kind == "prune":
        return dict(bytes=int(b + 8 * n), flops=int(2 * m))
    edges = m if kind == "unpruned" or not case.get("prune", True) else _core_edges(case)
    passes = 20 if kind == "certify" else case["passes"]
    if kind == "warm":
        b += 4 * edges
    return dict(bytes=int(b), flops=int(8 * edges * passes + 2 * m))


# ------------------------------------------------------------------ the same in 64-bit arithmetic

def _prune64(n, u, v, units):
    """Algorithm 2 in integers: (removal round per node, -1 kept; nodes ordered by first degree)."""
    dev = u.device
    rr = torch.full((n,), -1, dtype=torch.int64, device=dev)
    first = None
    r = 0
    while True:
        d = torch.zeros(n, dtype=torch.int64, device=dev).index_add_(0, u, units).index_add_(0, v, units)
        if first is None:
            first = d
        alive = rr < 0
        total, size = int(units.sum()), int(alive.sum())
        # d * size < total, without overflow: d < ceil(total / size)
        out = alive & (d < -(-total // max(size, 1)))
        r += 1
        if not bool(out.any()):
            break
        rr[out] = r
        keep = ~(out[u] | out[v])
        u, v, units = u[keep], v[keep], units[keep]
    return rr, torch.sort(first, stable=True).indices, r


def _fmix32(x):
    x = x.astype(np.uint32)
    x ^= x >> np.uint32(16)
    x *= np.uint32(0x85EBCA6B)
    x ^= x >> np.uint32(13)
    x *= np.uint32(0xC2B2AE35)
    x ^= x >> np.uint32(16)
    return x


def _colours(n, u, v, level):
    if not level:
        P = n + (n & 1) - 1
        return np.where(v == P, 2 * u, u + v) % max(P, 1)
    d = np.bincount(u, minlength=n) + np.bincount(v, minlength=n)
    order = np.lexsort((_fmix32(np.arange(u.shape[0])), np.minimum(d[u], d[v]), np.maximum(d[u], d[v])))
    last = [0] * n
    col = [0] * u.shape[0]
    for e, a, b in zip(order.tolist(), u[order].tolist(), v[order].tolist()):
        c = last[a] if last[a] >= last[b] else last[b]
        col[e] = c
        last[a] = last[b] = c + 1
    return np.asarray(col)


def _replay(n, u, v, w, s, passes, colour):
    """Algorithm 1's passes, class by class.  Returns (loads, splits)."""
    order = np.argsort(colour, kind="stable")
    cuts = np.flatnonzero(np.diff(colour[order])) + 1
    bounds = np.concatenate([[0], cuts, [order.shape[0]]]).tolist()
    a, b, w, s = u[order], v[order], w[order], s[order]
    l = np.bincount(a, weights=s, minlength=n) + np.bincount(b, weights=w - s, minlength=n)
    segs = [(a[x:y], b[x:y], w[x:y], s[x:y]) for x, y in zip(bounds[:-1], bounds[1:]) if y > x]
    for _ in range(passes):
        for ca, cb, cw, cs in segs:
            la, lb = l[ca], l[cb]
            d = np.maximum(np.minimum((la - lb) * 0.5, cs), cs - cw)
            l[ca] = la - d
            l[cb] = lb + d
            cs -= d
    out = np.empty_like(s)
    out[order] = s
    return l, out


def _best_prefix(n, u, v, w, loads):
    """The densest prefix of the load order (descending; the larger set on a tie): its density."""
    order = np.lexsort((-np.arange(n), -loads))
    pos = np.empty(n, np.int64)
    pos[order] = np.arange(n)
    W = np.cumsum(np.bincount(np.maximum(pos[u], pos[v]), weights=w, minlength=n))
    return float(np.max(W / np.arange(1, n + 1)))


def _features64(n, lo, hi, w):
    z = torch.zeros(n, dtype=torch.float64, device=lo.device)
    both, other = torch.cat([lo, hi]), torch.cat([hi, lo])
    w2 = torch.cat([w, w])
    d = z.index_add(0, both, w2)
    cnt = z.index_add(0, both, torch.ones_like(w2))
    sl = z.index_add(0, both, w2.log())
    two = z.index_add(0, both, d[other])
    return torch.stack([d.log1p(), sl / cnt.clamp(min=1), two.log1p()], 1), both, other, cnt


def _network64(p, n, lo, hi, w):
    """Splits and loads the network predicts (float64, nothing rounded)."""
    x, both, other, cnt = _features64(n, lo, hi, w)
    o = 0

    def take(k):
        nonlocal o
        o += k
        return p[o - k:o]
    W_in, b_in = take(192).view(3, 64), take(64)
    h = torch.relu(x @ W_in + b_in)
    for _ in range(3):
        W, b = take(8192).view(64, 128), take(64)
        m = torch.zeros_like(h).index_add(0, both, h[other]) / cnt.clamp(min=1)[:, None]
        h = torch.relu(torch.cat([h, m], 1) @ W.T + b)
    phi = h @ take(64)
    s = torch.sigmoid(phi[lo] - phi[hi]) * w
    return s, torch.zeros_like(x[:, 0]).index_add(0, lo, s).index_add(0, hi, w - s)


def _exact_batch(case, seed):
    gs = _batch_graphs(case, seed)
    cores, steps = [], 0
    for n, u, v in gs:
        tu, tv = torch.from_numpy(u).long(), torch.from_numpy(v).long()
        rr, _, rounds = _prune64(n, tu, tv, torch.ones_like(tu))
        keep = (rr < 0).numpy()
        cores.append((n, keep, rounds))
        steps += int(keep.sum()) * case["passes"]
        if steps > EXACT_STEPS:
            return None
    loads, rho = [], []
    for (n, u, v), (_, keep, _) in zip(gs, cores):
        new = np.cumsum(keep) - 1
        ke = keep[u] & keep[v]
        k, cu, cv = int(keep.sum()), new[u[ke]], new[v[ke]]
        w = np.ones(cu.shape[0])
        l, _ = _replay(k, cu, cv, w, 0.5 * w, case["passes"], _colours(k, cu, cv, False))
        full = np.zeros(n)
        full[keep] = l
        loads.append(full)
        rho.append(_best_prefix(k, cu, cv, w, l))
    return dict(rho=np.array(rho), S_size=None, in_S=None, n_core=None, m_core=None, rounds=None, status=None,
                loads=np.concatenate(loads))


def _exact_train(case, seed):
    n, lo, hi, t, params = _train_batch(case, seed)
    lo, hi = (torch.from_numpy(x).long().cuda() for x in (lo, hi))
    t = torch.from_numpy(t).double().cuda()
    p = torch.from_numpy(params).double().cuda().requires_grad_(True)
    _, loads = _network64(p, n, lo, hi, torch.ones(lo.shape[0], dtype=torch.float64, device="cuda"))
    loss = ((loads - t) ** 2).sum() / (t * t).sum()
    g, = torch.autograd.grad(loss, p)
    # Adam's first step: the bias-corrected moments are g and g^2
    new = p.detach() - 1e-3 * g / (g.abs() + 1e-8)
    return dict(loss=float(loss), grad=g.cpu().numpy(), loads=loads.detach().cpu().numpy(), params=new.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "certify":
        return None
    n, (u, v, w), _ = _graph(case, seed)
    u, v = u.long(), v.long()
    units = torch.ones_like(u) if w is None else torch.round(w.double() * GRID).long()
    out = {}
    keep = None
    if kind in ("prune", "warm") or case.get("prune"):
        rr, order, rounds = _prune64(n, u, v, units)
        out.update(kept=None, kept_edges=None, rounds=None)
        if kind == "prune":
            out.update(order=order.cpu().numpy(), removal_round=rr.cpu().numpy())
        keep = rr < 0
        new = torch.cumsum(keep, 0) - 1
        ke = keep[u] & keep[v]
        u, v, units = new[u[ke]], new[v[ke]], units[ke]
        n_cur = int(keep.sum())
    else:
        n_cur = n
    wt = units.double() / (1 if w is None else GRID)
    passes = 0 if kind == "prune" else case["passes"]
    if kind == "unpruned" and (case["hub_stars"] or u.shape[0] > EXACT_LEVEL_EDGES):
        return None
    level = kind == "unpruned" or n_cur > 53248
    if passes and n_cur * passes > EXACT_STEPS and not (level and u.shape[0] <= EXACT_LEVEL_EDGES):
        return None
    s = 0.5 * wt
    if kind == "warm":
        p = torch.from_numpy(warmstart.load_params()).double().cuda()
        s, _ = _network64(p, n_cur, u, v, wt)
        start = torch.zeros(n, dtype=torch.float64, device=u.device)
        ids = torch.nonzero(keep)[:, 0]
        start.index_add_(0, ids[u], s).index_add_(0, ids[v], wt - s)
        out["start_loads"] = start.cpu().numpy()
    if kind == "prune":
        # no pass has run: the extraction orders the core's nodes by their equal-split loads
        loads = (torch.zeros(n_cur, dtype=torch.float64, device=u.device).index_add_(0, u, s).index_add_(0, v, s)).cpu().numpy()
        uu, vv, ww = u.cpu().numpy(), v.cpu().numpy(), wt.cpu().numpy()
    else:
        uu, vv, ww, s = (x.cpu().numpy() for x in (u, v, wt, s))
        col = _colours(n_cur, uu, vv, level)
        if int(col.max(initial=0)) * passes > EXACT_STEPS:
            return None
        loads, _ = _replay(n_cur, uu, vv, ww, s, passes, col)
        out.update(sum_load_sq=float(np.sum(loads * loads)), max_load=float(loads.max()))
    full = np.zeros(n)
    full[keep.cpu().numpy() if keep is not None else slice(None)] = loads
    out.update(S=None, rho=_best_prefix(n_cur, uu, vv, ww, loads), loads=full)
    return out
