"""The paths a forward's kernels choose by size, at the sizes where they
switch or leave remainders, against the oracle (rules in gpu_helpers.py)."""
import numpy as np
import pytest
import torch

import workloads
from gpu_helpers import assert_parity, compare, make_layer, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def small(dtype="bf16", **kw):
    base = dict(tokens=300, d_model=128, d_ff=512, n_experts=4, n_blocks=4)
    base.update(kw)
    return workloads.spec("tiny_f32" if dtype == "f32" else "vit_s").with_(**base)


@pytest.mark.parametrize("T", [197, 1576, 5003])
def test_expert_tiles_split_over_chunks(T):
    """Fewer expert tiles than CTA pairs (T = 197, 1,576), or one and a half
    per pair (5,003): the tiles' chunks are split over the pairs, each part
    adding its partial sum."""
    wl = workloads.make_workload(workloads.spec("vit_s", tokens=T))
    assert_parity(wl, *_run(wl))


def _run(wl):
    g = run_gpu(wl)
    return g, compare(wl, g)
