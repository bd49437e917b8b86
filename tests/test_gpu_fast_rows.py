"""What the asynchronous kernels decide, rows at the edges of every kernel and table.  From a given
membership only three hubs have an improving move, each among communities that no other touches, so one
iteration has one outcome whatever the order: every hub in the best community of Eq. 2, ties to the
smaller id, everything else where it was.  A hub's neighbours lie in as many communities as it has arcs
(the fullest table), or two in each."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
from test_gpu_sweep import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def case(degrees, both, seed):
    """Hubs over pairs of vertices joined by an edge of weight 1000: a hub meets one member of each pair, or
    (`both`) the two.  (graph, start membership, membership after one iteration)"""
    rng = np.random.default_rng(seed)
    edges, weights, start, n = [], [], list(range(len(degrees))), len(degrees)
    for h, d in enumerate(degrees):
        left = d
        while left:
            k = 2 if both and left > 1 else 1
            edges += [(n, n + 1)] + [(h, n + j) for j in range(k)]
            weights += [1000] + [int(x) for x in rng.integers(1, 9, k)]
            start += [n, n]
            left -= k
            n += 2
    g = gg.from_edges(n, edges, weights=weights)
    start = np.array(start, dtype=np.int32)
    src = np.repeat(np.arange(n), np.diff(g.offsets))
    w = g.weights.astype(np.int64)
    k = np.bincount(src, w, n).astype(np.int64)
    two_m = int(k.sum())
    sigma = np.bincount(start, k, n).astype(np.int64)
    end = start.copy()
    for h in range(len(degrees)):  # K_h->d = 0 and Sigma_d = K_h: the hub is alone
        row = slice(g.offsets[h], g.offsets[h + 1])
        c, at = np.unique(start[g.targets[row]], return_inverse=True)
        kic = np.bincount(at, w[row]).astype(np.int64)
        score = two_m * kic - k[h] * sigma[c]
        best = int(np.argmax(score))  # the first of the largest: the smallest id
        if score[best] > 0:
            end[h] = c[best]
    # no member of a pair gains by joining a hub (8 against 1000 of weight, whatever has joined it)
    hubs = len(degrees)
    gain = two_m * (8 - 1000) - k[hubs:] * (k[:hubs].min() - (2100 + k[:hubs].max()))
    assert gain.max() < 0 and (end[:hubs] != start[:hubs]).all()
    return g, start, end


def canonical(m):
    return np.unique(m, return_inverse=True)[1].astype(np.int32)


@pytest.mark.parametrize("d", [4, 16, 128, 512, 2048, 4096, 9000])
@pytest.mark.parametrize("both", [False, True])
@pytest.mark.parametrize("tf", [1, 2, 4])
def test_hubs_take_their_best_community(cuda_ok, d, both, tf):
    import paper_2312_04876_gb300 as lv
    g, start, end = case([d - 1, d, d + 1], both, d + tf)
    L = lv.Louvain(0)
    for w in (g.weights, (g.weights / 8).astype(np.float32)):  # every sum is exact
        for profile in (0, 1):
            mem, r = L.run_from(*dev(g, w), torch.from_numpy(start).cuda(), mode="fast", fast_sync_small=1,
                                max_passes=1, max_iterations=1, table_factor=tf, profile=profile)
            assert np.array_equal(mem.cpu().numpy(), canonical(end))
            assert r.stats[0]["moves"] == 3
    L.close()
