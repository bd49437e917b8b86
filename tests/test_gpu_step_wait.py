"""Class steps whose bounded wait runs out, the colouring's not: at each of a launch's first barriers, so
in every part of a step -- between the insertion of a giant row's arcs into the shared tables and their
scan among them.  The call returns
LOUVAIN_ERR_TIMEOUT or the oracle's result, and whatever ran out, the next calls on the handle give the
oracle's result: the same graph, a smaller one whose giant rows use the same tables, an aggregation."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from test_gpu_sweep import dev, hubs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BARRIERS = list(range(24)) + [40, 10 ** 6]


@pytest.mark.parametrize("fp", [False, True])
def test_handle_is_usable_after_the_class_steps_time_out(cuda_ok, fp):
    import paper_2312_04876_gb300 as lv
    big = hubs([60000, 45000, 30000, 12000, 8193, 5000, 900, 200], 120000, 3, extra=0.5)
    small = hubs([15000, 9000, 700], 20000, 4, extra=0.5)
    cases = []
    for g in (big, small):
        w = (g.weights / 8).astype(np.float32) if fp else g.weights  # every sum is exact
        cases.append((g, w, oracle.louvain(g.offsets, g.targets, w, oracle.default_params())))
    L = lv.Louvain(0)

    def check(k):
        g, w, (ref, ref_q, ref_p, _) = cases[k]
        mem, r = L.run(*dev(g, w), mode="deterministic")
        assert np.array_equal(mem.cpu().numpy(), ref) and r.passes == ref_p and abs(r.modularity - ref_q) <= 1e-12

    ran_out = 0
    g, w, (ref, _, _, _) = cases[0]
    member = np.arange(small.n, dtype=np.int32) % 3  # three communities of more than 8192 arcs each
    for k, barrier in enumerate(BARRIERS):
        L.inject_step_wait(1, barrier)
        try:
            mem, _ = L.run(*dev(g, w), mode="deterministic")
            assert np.array_equal(mem.cpu().numpy(), ref)
        except lv.LouvainError as e:
            assert e.status == 4 and "local-moving" in str(e)  # LOUVAIN_ERR_TIMEOUT
            ran_out += 1
        L.inject_step_wait(0)
        if k % 3 == 2:  # the merge is the next user of the tables
            o, t, aw = L.aggregate(*dev(small, cases[1][1]), torch.from_numpy(member).cuda(), 3)
            rows = np.repeat(np.arange(3), np.diff(o.cpu().numpy()))
            got = np.zeros((3, 3))
            np.add.at(got, (rows, t.cpu().numpy()), aw.cpu().numpy())
            want = np.zeros((3, 3))
            at = np.repeat(np.arange(small.n), np.diff(small.offsets))
            np.add.at(want, (member[at], member[small.targets]), cases[1][1])
            assert np.array_equal(got, want)
        check(k % 2)
        check((k + 1) % 2)
    assert ran_out >= 1
    L.close()
