"""Scans and counting sorts at the sizes where their launches change: one block, tiles whose blocks sum
the tiles before them, tiles with a prefix launch between; sorts by one block and by many."""
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


@pytest.mark.parametrize("n", [0, 1, 3, 5, 127, 4095, 4096, 4097, 32767, 32768, 32769, 2048 * 4096, 2048 * 4096 + 1])
def test_scan_sizes_both_entry_points(L, n):
    import paper_2312_04876_gb300 as lv
    x = np.random.default_rng(n).integers(-(1 << 40), 1 << 40, size=n, dtype=np.int64)
    ref = np.concatenate([[0], np.cumsum(x)])
    d = torch.from_numpy(x).cuda()
    for out, tot in (L.exclusive_scan(d), lv.exclusive_scan_static(d)):
        assert np.array_equal(out.cpu().numpy(), ref) and tot == ref[-1]
    buf = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    buf[:n] = d
    lv.exclusive_scan_static(buf[:n], buf)  # in place
    assert np.array_equal(buf.cpu().numpy(), ref)


@pytest.mark.parametrize("mode", ["deterministic", "fast"])
@pytest.mark.parametrize("n", [2, 1023, 1025, 8191, 8192, 8193])
def test_runs_around_the_one_block_sort(L, n, mode):
    # isolated vertices and hubs of every degree bucket among them
    rng = np.random.default_rng(n)
    e = {(0, 1)} | {(0, int(v)) for v in range(1, n, 2)} | {(1, int(v)) for v in rng.integers(2, max(n, 3), n // 9) if v < n}
    e |= {(int(min(a, b)), int(max(a, b))) for a, b in rng.integers(0, n, (n // 2, 2)) if a != b}
    g = gg.from_edges(n, sorted(e))
    mem, r = L.run(*(torch.from_numpy(x).cuda() for x in (g.offsets, g.targets, g.weights)), mode=mode)
    mem = mem.cpu().numpy()
    if mode == "deterministic":
        ref, ref_q, _, _ = oracle.louvain(g.offsets, g.targets, g.weights, oracle.default_params())
        assert np.array_equal(mem, ref) and r.modularity == ref_q
    assert abs(oracle.modularity(g.offsets, g.targets, g.weights, mem) - r.modularity) <= 1e-12
