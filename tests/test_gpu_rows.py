"""The per-bucket and giant-row kernels at the edges of their rows (4, 16, 128, 512, 2048, 4096 arcs) and of
their tables (1, 2 and 4 slots a key).  A profiled deterministic run takes its class steps through
them, one launch a bucket: memberships and modularity equal the oracle's exactly.  Fast runs take them
asynchronously: the result is a partition whose modularity is the one returned."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from test_gpu_sweep import dev, hubs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L(cuda_ok):
    import paper_2312_04876_gb300 as lv
    h = lv.Louvain(0)
    yield h
    h.close()


@pytest.mark.parametrize("d", [4, 16, 128, 512, 2048, 4096, 9000])
@pytest.mark.parametrize("tf", [1, 2, 4])
def test_rows_at_bucket_edges(L, d, tf):
    g = hubs([d - 1, d, d + 1], max(60, 3 * d), d + tf, extra=1.0)
    ref, ref_q, ref_p, _ = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params())
    mem, r = L.run(*dev(g), mode="deterministic", profile=1, table_factor=tf)
    assert np.array_equal(mem.cpu().numpy(), ref) and r.modularity == ref_q and r.passes == ref_p
    for profile in (0, 1):
        mem, r = L.run(*dev(g), mode="fast", fast_sync_small=1, profile=profile, table_factor=tf)
        q = oracle.modularity(g.offsets, g.targets, g.weights, mem.cpu().numpy())
        assert abs(q - r.modularity) <= 1e-12


@pytest.mark.parametrize("over", [dict(pruning=0), dict(giant_min_degree=2048), dict(lm_blocks_per_sm=1)])
def test_controls_and_float_weights(L, over):
    g = hubs([20000, 6000, 2500, 900, 300, 100, 10], 40000, 5)
    w = (g.weights / 8).astype(np.float32)  # every sum is exact
    ref_over = {k: v for k, v in over.items() if k == "pruning"}
    for wt in (g.weights, w):
        ref, ref_q, _, _ = oracle.louvain(g.offsets, g.targets, wt, oracle.default_params(**ref_over))
        mem, r = L.run(*dev(g, wt), mode="deterministic", profile=1, **over)
        assert np.array_equal(mem.cpu().numpy(), ref) and abs(r.modularity - ref_q) <= 1e-12
