"""Validation of the input graph where its arc-parallel check can go wrong: runs of empty rows longer
than a warp, hubs over many warps' ranges, tiny graphs, and a single bad target, weight or missing
mirror arc at the first, a middle and the last arc.  What the oracle's definition accepts runs, the rest
is refused before anything else reads it."""
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


def spread(n, ids, edges):
    """The edges over ids mapped to vertices far apart: long runs of empty rows between them."""
    return gg.from_edges(n, [(int(ids[a]), int(ids[b])) for a, b in edges])


def ring(k):
    return [(i, (i + 1) % k) for i in range(k)]


GRAPHS = {
    "pair": lambda: gg.from_edges(2, [(0, 1)]),
    "loop_only": lambda: gg.from_edges(3, [(1, 1)]),
    "empty_runs": lambda: spread(5000, np.r_[0, 33, 66, 98, 1000, 1032, 4967, 4999], ring(8)),
    "all_at_the_end": lambda: spread(3000, np.arange(2960, 3000), ring(40)),
    "star_30000": lambda: gg.from_edges(30001, [(0, i) for i in range(1, 30001)]),
    "hub_at_the_end": lambda: gg.from_edges(20001, [(20000, i) for i in range(0, 20000, 2)] + [(i, i + 1) for i in range(0, 9000, 3)]),
    "sbm": lambda: gg.sbm(3001, 30, 0.1, 0.002, 3),
}


def run(L, g, t, w):
    return L.run(*(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (g.offsets, t, w)), mode="deterministic",
                 validate=1)


@pytest.mark.parametrize("fp", [False, True])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_accepts_and_refuses(L, name, fp):
    import paper_2312_04876_gb300 as lv
    g = GRAPHS[name]()
    w = (g.weights / 4).astype(np.float32) if fp else g.weights
    ref, _, _, _ = oracle.louvain(g.offsets, g.targets, w, oracle.default_params())
    assert np.array_equal(run(L, g, g.targets, w)[0].cpu().numpy(), ref)
    bad_weights = [0, -1] + ([np.inf, np.nan] if fp else [])
    rows = np.repeat(np.arange(g.n), np.diff(g.offsets))
    for at in sorted({0, g.n_arcs // 3, g.n_arcs // 2, g.n_arcs - 1}):
        for bad in (-1, g.n):
            t = g.targets.copy()
            t[at] = bad
            with pytest.raises(lv.LouvainError, match="target"):
                run(L, g, t, w)
        for bad in bad_weights:
            x = w.copy()
            x[at] = bad
            with pytest.raises(lv.LouvainError, match="weight"):
                run(L, g, g.targets, x)
        if g.targets[at] != rows[at]:
            x = w.copy()
            x[at] += 1
            with pytest.raises(lv.LouvainError, match="symmetric"):
                run(L, g, g.targets, x)
