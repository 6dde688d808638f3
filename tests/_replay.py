"""Algorithm 1's passes in the circle colouring's order, replayed in FP32 with numpy, operation for
operation: what every pass kernel of schedule 1 computes, to the bit.

The initial loads are FP64 sums of the splits; `grid_splits` gives splits whose sums are exact, so
that they do not depend on the order of the additions.
"""
import numpy as np

F = np.float32


def grid_splits(m, w, seed):
    """Uneven splits in [0, w_e], multiples of 2^-16 (sums of them are exact in FP64)."""
    r = np.random.default_rng(seed).random(m)
    lim = np.ones(m) if w is None else w.astype(np.float64)
    return (np.floor(r * lim * 65536.0) / 65536.0).astype(F)


def classes(n, u, v):
    """Edge ids of every colour class of the circle method, in the order of the colours."""
    P = n + (n & 1) - 1
    a, b = u.astype(np.int64), v.astype(np.int64)
    c = np.where((n & 1 == 0) & (b == n - 1), 2 * a, a + b) % P
    order = np.argsort(c, kind="stable")
    heads = np.flatnonzero(np.diff(c[order], prepend=-1))
    return np.split(order, heads[1:])


def replay(n, u, v, w, s0, passes, pair):
    """Splits after `passes` passes from the splits s0: pair loads (two FP32) or single FP32 ones."""
    wt = np.ones(u.shape[0], F) if w is None else w.astype(F)
    s = s0.astype(F).copy()
    l64 = (np.bincount(u, weights=s.astype(np.float64), minlength=n) +
           np.bincount(v, weights=wt.astype(np.float64) - s.astype(np.float64), minlength=n))
    hi = l64.astype(F)
    lo = (l64 - hi.astype(np.float64)).astype(F)
    if not pair:
        hi, lo = hi + lo, np.zeros(n, F)
    cl = classes(n, u, v)
    for _ in range(passes):
        for e in cl:
            a, b = u[e], v[e]
            ax, bx = hi[a], hi[b]
            diff = (ax - bx) + (lo[a] - lo[b]) if pair else ax - bx
            se, we = s[e], wt[e]
            dd = np.minimum(np.maximum(diff * F(0.5), se - we), se)
            ta, tb = ax - dd, bx + dd
            if pair:   # Knuth's TwoSum
                ba, bb = ta - ax, tb - bx
                lo[a] += (ax - (ta - ba)) + (-dd - ba)
                lo[b] += (bx - (tb - bb)) + (dd - bb)
            hi[a], hi[b] = ta, tb
            s[e] = np.minimum(se - dd, we)
    return s
