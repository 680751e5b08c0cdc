"""GPU tests of what a caller may do around the calls: options set for another call, a sharded
step that is dropped, kernels of the caller's own ahead of a step, buffers side by side."""
import numpy as np
import pytest
import torch

from paper_2603_18112_gb300 import tula_ags as T
from paper_2603_18112_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_18112_gb300 import build
    build.build()
    T.lib()


def _normal_pset(sizes):
    ps = W.ParamSet("sizes")
    for n in sizes:
        ps.add((int(n),), W.KIND_NORMAL)
    return ps


def _workload(seed):
    return W.workload("stress_k4", seed=seed, factor_range=(0.1, 10.0), zero_patterns=False)


@pytest.mark.parametrize("gran", [T.TULA_SCALE_PER_TENSOR, T.TULA_SCALE_PER_ELEMENT])
def test_update_scale_leaves_the_statistics_alone(gran):
    """tula_ags_update_scale with the options of a step, whose layer_stats is set: the rows are
    the step's and stay as they are."""
    wl = _workload(301)
    buf = W.allocate(wl, "cuda", K=2, pset=_normal_pset((1, 5, 1000, 20000)))
    W.fill_state(buf, wl)
    W.fill_grads(buf, wl, step=1)
    elem = [torch.ones_like(t) for t in buf.w]
    st = T.AGSOptimizerStep(buf.w, buf.g, buf.m, scale_elem=elem)
    st.step(wl.lr, wl.momentum, wl.weight_decay)
    rows = st.stats.clone()
    st.hp.granularity = gran
    T.tula_ags_update_scale(buf.g[1], buf.g[0], st.hp)
    torch.cuda.synchronize()
    assert torch.equal(st.stats, rows)
    changed = elem if gran == T.TULA_SCALE_PER_ELEMENT else [st.scale]
    assert all(bool((t != 1).any()) for t in changed)
