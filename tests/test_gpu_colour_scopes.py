"""The persistent colouring at the sizes where its paths change: one block, one cluster and the grid;
8- and 32-arc list entries; rows at the edges of a chunk, of what a block keeps and of the bitmap
words; more ready vertices than a block keeps.  Colours equal the oracle's exactly."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L(cuda_ok):
    import paper_2312_04876_gb300 as lv
    h = lv.Louvain(0)
    yield h
    h.close()


def clique(k, base=0):
    return [(base + i, base + j) for i in range(k) for j in range(i)]


def random_edges(n, m, seed):
    e = np.random.default_rng(seed).integers(0, n, size=(m, 2))
    e = e[e[:, 0] != e[:, 1]]
    return np.unique(np.sort(e, axis=1), axis=0)


def from_edges(n, e):
    return gg.from_edges(n, [tuple(map(int, x)) for x in e])


CASES = {
    # chunk edges: degree 8 / 9 (8-arc entries), 31 / 32 / 33 (bitmap words, 32-arc entries), 128 / 129
    # (the longest rows a block keeps)
    **{f"clique{k}": (lambda k=k: from_edges(k, clique(k))) for k in (2, 9, 10, 32, 33, 34, 129, 130)},
    "cluster_clique350": lambda: from_edges(350, clique(350)),
    "star_5000": lambda: from_edges(5000, [(0, i) for i in range(1, 5000)]),
    # more ready vertices than a block keeps, one block: 8-arc and 32-arc entries
    "pairs_8000": lambda: from_edges(8000, [(2 * i, 2 * i + 1) for i in range(4000)]),
    "pairs_and_clique": lambda: from_edges(4540, clique(140) + [(140 + 2 * i, 141 + 2 * i) for i in range(2200)]),
    # the grid: low degree and ordinary, isolated vertices among them
    "grid_low": lambda: from_edges(40003, random_edges(40003, 45000, 1)),
    "grid_mid": lambda: from_edges(20011, random_edges(20011, 200000, 2)),
    # many rows of 513-2048 arcs (a warp each) and hubs
    "dense_2000": lambda: from_edges(2000, random_edges(2000, 900000, 3)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_colouring_paths_match_oracle(L, name):
    g = CASES[name]()
    o, t = torch.from_numpy(g.offsets).cuda(), torch.from_numpy(g.targets).cuda()
    for seed in (0, 7):
        col, nc = L.colour(o, t, seed, 1)
        ref, ref_nc = oracle.colour(g.offsets, g.targets, seed, 1)
        assert nc == ref_nc and np.array_equal(col.cpu().numpy(), ref)


def test_colouring_counts_repeated_arcs_and_loops(L):
    """Repeated arcs count once per copy on both sides; self-loops not at all."""
    rng = np.random.default_rng(5)
    n = 200
    e = rng.integers(0, n, size=(3000, 2))
    src = np.concatenate([e[:, 0], e[e[:, 0] != e[:, 1], 1]])
    dst = np.concatenate([e[:, 1], e[e[:, 0] != e[:, 1], 0]])
    order = np.argsort(src, kind="stable")
    offsets = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    targets = dst[order].astype(np.int32)
    col, nc = L.colour(torch.from_numpy(offsets).cuda(), torch.from_numpy(targets).cuda(), 3, 0)
    ref, ref_nc = oracle.colour(offsets, targets, 3, 0)
    assert nc == ref_nc and np.array_equal(col.cpu().numpy(), ref)
