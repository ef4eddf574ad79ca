"""Clouds with long neighbour lists (not a test): each point's neighbours and
theirs, 25 to 60 of them, so that points have more than 32 neighbours earlier
or later in the sweep order, which the packed sweeps do not take."""
import copy

import numpy as np


def two_rings(cloud, keep=255):
    """The cloud with neighbour lists of two rings (at most `keep`, nearest first)."""
    off, idx = np.asarray(cloud.nbr_off), np.asarray(cloud.nbr_idx)
    x, y = np.asarray(cloud.x), np.asarray(cloud.y)
    lists = []
    for p in range(cloud.n):
        one = idx[off[p]:off[p + 1]]
        far = np.setdiff1d(np.concatenate([idx[off[i]:off[i + 1]] for i in one]), np.append(one, p))
        far = far[np.argsort((x[far] - x[p]) ** 2 + (y[far] - y[p]) ** 2, kind="stable")]
        lists.append(np.concatenate([one, far])[:keep])
    c = copy.copy(cloud)
    c.nbr_off = np.concatenate([[0], np.cumsum([len(t) for t in lists])]).astype(np.int32)
    c.nbr_idx = np.concatenate(lists).astype(np.int32)
    return c


def longest_list(cloud, order):
    """Longest list of earlier or later neighbours in the sweep order (order[t] = point at position t)."""
    pos = np.empty(cloud.n, np.int64)
    pos[order] = np.arange(cloud.n)
    off, idx = np.asarray(cloud.nbr_off), np.asarray(cloud.nbr_idx)
    best = 0
    for p in range(cloud.n):
        d = pos[idx[off[p]:off[p + 1]]] < pos[p]
        best = max(best, int(d.sum()), int((~d).sum()))
    return best
