"""The reweighting decode finds shortest paths by relaxing every node until nothing changes and then
names predecessors.  This checks, on random graphs full of ties, that distances and parities are those
of Dijkstra's algorithm with nodes popped in (distance, index) order, each node's edges relaxed in
(neighbour, observable) order, predecessors changed only on a strict improvement and the boundary a
sink (numpy FP64 on both sides)."""
import heapq
import math

import numpy as np
import pytest


def _graph(rng, n, ties):
    """Adjacency lists over nodes 0..n (n = boundary), entries (neighbour, obs, weight) sorted."""
    edges = []
    for u in range(n):
        for v in rng.choice(n + 1, size=3, replace=False):
            if v != u:
                edges.append((u, int(v)))
    edges += edges[: n // 3]  # parallel edges
    adj = [[] for _ in range(n + 1)]
    for q, (u, v) in enumerate(edges):
        w = float(rng.integers(1, 4)) if ties else float(rng.exponential(1.0)) + 2.0 ** -20
        ob = int(rng.integers(0, 2))
        adj[u].append((v, ob, q, w))
        adj[v].append((u, ob, q, w))
    return [sorted(a) for a in adj]


def _dijkstra(adj, n, src):
    dist = [math.inf] * (n + 1)
    par = [0] * (n + 1)
    done = [False] * (n + 1)
    dist[src] = 0.0
    heap = [(0.0, src)]
    while heap:
        d, u = heapq.heappop(heap)
        if done[u] or d != dist[u]:
            continue
        done[u] = True
        if u == n:
            continue
        for v, ob, _, w in adj[u]:
            nd = d + w
            if nd < dist[v]:
                dist[v] = nd
                par[v] = par[u] ^ ob
                heapq.heappush(heap, (nd, v))
    return dist, par


def _relax(adj, n, src):
    dist = [math.inf] * (n + 1)
    dist[src] = 0.0
    again = True
    while again:  # nodes 0..n-1, from neighbours other than the boundary
        again = False
        for v in range(n):
            best = min([dist[v]] + [dist[u] + w for u, _, _, w in adj[v] if u != n])
            if best < dist[v]:
                dist[v] = best
                again = True
    pred = [None] * (n + 1)
    for v in range(n + 1):
        best, du = (math.inf if v == n else dist[v]), math.inf
        for u, ob, _, w in adj[v]:
            if u == n:
                continue
            nd = dist[u] + w
            if nd != math.inf and ((v == n and nd < best) or (nd == best and dist[u] < du)):
                best, du, pred[v] = nd, dist[u], (u, ob)
        if v == n:
            dist[n] = best
    pred[src] = None
    par = []
    for v in range(n + 1):
        p, e = 0, pred[v]
        while e is not None:
            p ^= e[1]
            e = pred[e[0]]
        par.append(p)
    return dist, par


@pytest.mark.parametrize("ties", [True, False])
def test_relaxation_equals_dijkstra(ties):
    rng = np.random.default_rng(5 + ties)
    for _ in range(60):
        n = int(rng.integers(2, 40))
        adj = _graph(rng, n, ties) if n >= 3 else [[(1, 0, 0, 1.0), (2, 1, 1, 1.0)], [(0, 0, 0, 1.0)], [(0, 1, 1, 1.0)]]
        for src in range(n):
            assert _dijkstra(adj, n, src) == _relax(adj, n, src)
