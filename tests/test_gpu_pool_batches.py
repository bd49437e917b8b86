"""Classes with more giant rows in the shared tables (over 8192 arcs) than a step takes at once: 32, 33, 64
and 65 of them -- one batch full, one over, two full, one over -- and 70 whose communities change over
several iterations.  Memberships, modularity, passes and iterations equal the oracle's exactly, on the
grid and on one block."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def stars(hubs, extra, seed):
    """Hubs of 8193 leaves and more, disjoint, and `extra` random edges among the leaves."""
    rng = np.random.default_rng(seed)
    size = 8193 + rng.integers(0, 300, hubs)
    n = hubs + int(size.sum())
    a, b = rng.integers(hubs, n, (2, extra))
    e = np.concatenate([np.stack([np.repeat(np.arange(hubs), size), np.arange(hubs, n)], 1),
                        np.stack([np.minimum(a, b), np.maximum(a, b)], 1)[a != b]])
    e = np.unique(e, axis=0)
    w = rng.integers(1, 9, len(e)).astype(np.int32)
    src, dst = np.concatenate([e[:, 0], e[:, 1]]), np.concatenate([e[:, 1], e[:, 0]])
    order = np.argsort(src, kind="stable")
    offsets = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    return offsets, dst[order].astype(np.int32), np.concatenate([w, w])[order]


@pytest.mark.parametrize("hubs,extra,in_class", [(32, 0, 32), (33, 0, 33), (64, 0, 64), (65, 0, 65), (70, 5000, 33)])
@pytest.mark.parametrize("fp", [False, True])
def test_giants_of_a_class_in_batches(cuda_ok, hubs, extra, in_class, fp):
    import paper_2312_04876_gb300 as lv
    offsets, targets, w = stars(hubs, extra, 3)
    col, _ = oracle.colour(offsets, targets, 0, 0)
    assert np.bincount(col[:hubs]).max() >= in_class
    w = (w / 8).astype(np.float32) if fp else w  # every sum is exact
    ref, ref_q, ref_p, ref_s = oracle.louvain(offsets, targets, w, oracle.default_params())
    L = lv.Louvain(0)
    dev = [torch.from_numpy(x).cuda() for x in (offsets, targets, w)]
    for refused in (False, True):
        L.inject_launch_refusal(refused)
        mem, r = L.run(*dev, mode="deterministic")
        assert np.array_equal(mem.cpu().numpy(), ref) and r.passes == ref_p and abs(r.modularity - ref_q) <= 1e-12
        assert [s["iterations"] for s in r.stats] == [s["iterations"] for s in ref_s]
    L.close()
