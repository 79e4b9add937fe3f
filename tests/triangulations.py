"""Unimodular triangulations of d*Delta_2 that need not be regular, for tests:
any maximal set of primitive segments without crossings is one."""
from math import gcd

import numpy as np


def greedy_triangulation(d: int, seed: int, first=(), short: bool = False) -> np.ndarray:
    """(E, 4) int32 edges: the segments of `first` (rows i1, j1, i2, j2, free of
    crossings), then every primitive segment, in a random order or (short)
    shorter ones first, that crosses none before it."""
    pts = [(i, j) for j in range(d + 1) for i in range(d + 1 - j)]
    segs = np.array([p + q for n, p in enumerate(pts) for q in pts[n + 1:]
                     if gcd(abs(p[0] - q[0]), abs(p[1] - q[1])) == 1], dtype=np.int64)
    rng = np.random.default_rng(seed)
    segs = segs[rng.permutation(len(segs))]
    if short:
        len2 = (segs[:, 0] - segs[:, 2]) ** 2 + (segs[:, 1] - segs[:, 3]) ** 2
        segs = segs[np.argsort(len2, kind="stable")]
    segs = np.concatenate([np.array(first, dtype=np.int64).reshape(-1, 4), segs])

    def side(a, b, p):  # of points p, as seen from a towards b
        return np.sign((b[..., 0] - a[..., 0]) * (p[..., 1] - a[..., 1])
                       - (b[..., 1] - a[..., 1]) * (p[..., 0] - a[..., 0]))

    free = np.ones(len(segs), dtype=bool)  # crosses no chosen segment
    chosen, seen = [], set()
    a, b = segs[:, :2], segs[:, 2:]
    for n, s in enumerate(segs):
        key = tuple(sorted([tuple(s[:2].tolist()), tuple(s[2:].tolist())]))
        if not free[n] or key in seen:
            continue
        seen.add(key)
        chosen.append(s)
        p, q = s[None, :2], s[None, 2:]
        free &= ~((side(a, b, p) * side(a, b, q) < 0) & (side(p, q, a) * side(p, q, b) < 0))
    if len(chosen) != 3 * d * (d + 1) // 2:
        raise ValueError("the given segments cross")
    return np.array(chosen, dtype=np.int32)


def apex_triangulation(d: int, k: int, seed: int = 0) -> np.ndarray:
    """With the edge (0, d)-(k, 0), gcd(d, k) = 1: vertex (0, -d) of the
    reflected triangulation is next to the middle row."""
    return greedy_triangulation(d, seed, first=[(0, d, k, 0)], short=True)


def hub_triangulation(d: int, n: int, seed: int = 0) -> np.ndarray:
    """With the origin joined to n interior points (and (1, 0), (0, 1)): 4n + 3
    neighbours of the middle vertex (0, 0) come before it in the sweep."""
    inner = sorted((i + j, i, j) for i in range(1, d) for j in range(1, d - i) if gcd(i, j) == 1)
    if len(inner) < n:
        raise ValueError(f"degree {d} has {len(inner)} primitive interior points")
    return greedy_triangulation(d, seed, first=[(0, 0, i, j) for _, i, j in inner[:n]], short=True)
