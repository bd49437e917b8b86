"""The colouring and the class steps where the driver refuses a cluster or a cooperative grid: one block
takes every row of every kind, whatever grid the step records were made for.  Memberships, modularity,
passes and iterations equal the oracle's exactly, and again once launches are accepted."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle
from test_gpu_sweep import dev, hubs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRAPHS = {
    # the grid: rows of every kind, several pool giants
    "hubs": lambda: hubs([20000, 9000, 8193, 8192, 5000, 3000, 700, 200, 60], 40000, 11, extra=0.5),
    # a cluster: dense, many narrow steps, rows of two and of three kinds
    "dense_600": lambda: gg.sbm(600, 6, 0.5, 0.1, 5),
    "dense_2500": lambda: hubs([2300, 1500, 900, 700], 2500, 3, extra=20.0),
    # no long rows
    "sbm": lambda: gg.sbm(20000, 40, 0.02, 0.0005, 7),
    "low_degree": lambda: hubs([10, 8], 50000, 2, extra=1.2),
}


@pytest.fixture(scope="module")
def L(cuda_ok):
    import paper_2312_04876_gb300 as lv
    h = lv.Louvain(0)
    yield h
    h.close()


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("over", [dict(), dict(pruning=0, max_iterations=3), dict(wait_spins=1 << 22)])
def test_refused_grids_change_no_result(L, name, over):
    g = GRAPHS[name]()
    ref_over = {k: v for k, v in over.items() if k != "wait_spins"}
    ref, ref_q, ref_p, ref_s = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params(**ref_over))
    for refused in (True, False):
        L.inject_launch_refusal(refused)
        mem, r = L.run(*dev(g), mode="deterministic", **over)
        assert np.array_equal(mem.cpu().numpy(), ref) and r.modularity == ref_q and r.passes == ref_p
        assert [s["iterations"] for s in r.stats] == [s["iterations"] for s in ref_s]


def test_refused_grids_float_weights_batch_and_colours(L):
    graphs = [GRAPHS[k]() for k in ("dense_600", "hubs", "sbm")]
    vo = np.concatenate([[0], np.cumsum([g.n for g in graphs])])
    ao = np.concatenate([[0], np.cumsum([g.n_arcs for g in graphs])])
    o = np.concatenate([[0]] + [g.offsets[1:] + ao[k] for k, g in enumerate(graphs)])
    t, w = (np.concatenate([getattr(g, f) for g in graphs]) for f in ("targets", "weights"))
    w = (w / 8).astype(np.float32)  # every sum is exact
    L.inject_launch_refusal(True)
    mem, per, _ = L.run_batch(vo, *(torch.from_numpy(x).cuda() for x in (o, t, w)), mode="deterministic")
    mem = mem.cpu().numpy()
    for k, g in enumerate(graphs):
        ref, ref_q, ref_p, _ = oracle.louvain(g.offsets, g.targets, w[ao[k]:ao[k + 1]], oracle.default_params())
        assert np.array_equal(mem[vo[k]:vo[k + 1]], ref)
        assert abs(per[k]["modularity"] - ref_q) <= 1e-12 and per[k]["passes"] == ref_p
        col, nc = L.colour(*dev(g)[:2], 0, 1)
        ref_col, ref_nc = oracle.colour(g.offsets, g.targets, 0, 1)
        assert nc == ref_nc and np.array_equal(col.cpu().numpy(), ref_col)
    L.inject_launch_refusal(False)
