"""Autotuning times the grid cap of the local-moving kernels only where a run launches them: a deterministic
run without wide classes takes its class steps in one persistent launch, whose grid the cap does not change."""
from __future__ import annotations

import pytest

import graphgen as gg
from test_gpu_sweep import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_deterministic_autotuning_leaves_the_grid_cap_at_its_default(cuda_ok):
    import paper_2312_04876_gb300 as lv
    L = lv.Louvain(0)
    for seed in range(6):
        g = gg.sbm(3000, 30, 0.1, 0.002, seed)
        tuned, ms = L.autotune(*dev(g), mode="deterministic", reps=1)
        assert ms > 0.0 and tuned.lm_blocks_per_sm == 16
    L.close()
