"""The persistent class steps of the deterministic schedule at the sizes where their paths change: rows
at the edges of every group size (4, 16, 128, 512, 2048, 4096, 8192 arcs), giant rows in the shared
pool, steps with more vertices than a block keeps, pruning off, float weights with exact sums,
batches.  Memberships, modularity, passes and iterations equal the oracle's exactly."""
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


def dev(g, w=None):
    return tuple(torch.from_numpy(x).cuda() for x in (g.offsets, g.targets, g.weights if w is None else w))


def hubs(degrees, n, seed, extra=3.0):
    """Hubs of the given degrees over n vertices, plus a sparse random graph among all of them."""
    rng = np.random.default_rng(seed)
    e = set()
    for h, d in enumerate(degrees):
        for v in rng.choice(np.arange(len(degrees), n), size=d, replace=False):
            e.add((h, int(v)))
    m = int(extra * n)
    for a, b in zip(rng.integers(len(degrees), n, m), rng.integers(len(degrees), n, m)):
        if a != b:
            e.add((int(min(a, b)), int(max(a, b))))
    w = np.random.default_rng(seed + 1)
    return gg.from_edges(n, sorted(e), weights=[int(x) for x in w.integers(1, 9, len(e))])


def check(L, g, **over):
    ref, ref_q, ref_p, ref_s = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params(**over))
    mem, r = L.run(*dev(g), mode="deterministic", **over)
    assert np.array_equal(mem.cpu().numpy(), ref)
    assert r.modularity == ref_q and r.passes == ref_p
    assert [s["iterations"] for s in r.stats] == [s["iterations"] for s in ref_s]


@pytest.mark.parametrize("d", [4, 16, 128, 512, 2048, 4096, 8192])
def test_rows_at_group_edges(L, d):
    check(L, hubs([d - 1, d, d + 1], max(60, 3 * d), d, extra=1.0), seed=d)


def test_giants_of_both_kinds_in_one_class(L):
    # disjoint hubs share colour classes: block rows and pool rows decide in the same steps
    check(L, hubs([20000, 9000, 8192, 8193, 5000, 4097, 3000, 700], 60000, 11, extra=0.5))


@pytest.mark.parametrize("over", [dict(pruning=0), dict(giant_min_degree=2048), dict(max_iterations=1),
                                  dict(tolerance=0.0, max_iterations=7), dict(compact=0), dict(wait_spins=1 << 22)])
def test_controls(L, over):
    g = hubs([6000, 2500, 900, 300], 20000, 5)
    ref_over = {k: v for k, v in over.items() if k not in ("giant_min_degree", "compact", "wait_spins")}
    ref, ref_q, _, _ = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params(**ref_over))
    mem, r = L.run(*dev(g), mode="deterministic", **over)
    assert np.array_equal(mem.cpu().numpy(), ref) and r.modularity == ref_q


@pytest.mark.parametrize("n", [1300, 33000, 700000])
def test_steps_with_more_rows_than_a_block_keeps(L, n):
    # few colours on a long cycle with chords: hundreds to hundred thousands of vertices a step
    rng = np.random.default_rng(n)
    e = {(i, i + 1) for i in range(n - 1)} | {tuple(sorted(map(int, x))) for x in rng.integers(0, n, (n // 2, 2)) if x[0] != x[1]}
    check(L, gg.from_edges(n, sorted(e)))


def test_float_weights_with_exact_sums(L):
    g = hubs([9000, 3000, 600, 100], 30000, 9)
    w = (g.weights / 8).astype(np.float32)
    ref, ref_q, ref_p, _ = oracle.louvain(g.offsets, g.targets, w, oracle.default_params())
    mem, r = L.run(*dev(g, w), mode="deterministic")
    assert np.array_equal(mem.cpu().numpy(), ref) and r.passes == ref_p
    assert abs(r.modularity - ref_q) <= 1e-12


def test_batch_with_hubs_equals_each_graph_alone(L):
    graphs = [hubs([9000, 500], 20000, 1), gg.sbm(3000, 30, 0.1, 0.002, 3), hubs([40], 90, 2), hubs([5000, 4500], 12000, 4)]
    vo = np.concatenate([[0], np.cumsum([g.n for g in graphs])])
    ao = np.concatenate([[0], np.cumsum([g.n_arcs for g in graphs])])
    o = np.concatenate([[0]] + [g.offsets[1:] + ao[k] for k, g in enumerate(graphs)])
    t, w = (np.concatenate([getattr(g, f) for g in graphs]) for f in ("targets", "weights"))
    mem, per, _ = L.run_batch(vo, *(torch.from_numpy(x).cuda() for x in (o, t, w)), mode="deterministic")
    mem = mem.cpu().numpy()
    for k, g in enumerate(graphs):
        ref, ref_q, ref_p, _ = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params())
        assert np.array_equal(mem[vo[k]:vo[k + 1]], ref)
        assert abs(per[k]["modularity"] - ref_q) <= 1e-12 and per[k]["passes"] == ref_p
