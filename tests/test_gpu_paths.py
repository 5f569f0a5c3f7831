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


@pytest.mark.parametrize("shape", [
    dict(d_model=72, d_ff=60, n_blocks=4),     # M = 15: unaligned weight columns; d % 32 = 8
    dict(d_model=64, d_ff=280, n_blocks=4),    # M = 70: one whole 64-column item and 6 columns
    dict(d_model=200, d_ff=512, n_blocks=2),   # several reduction steps, d % 64 = 8
])
@pytest.mark.parametrize("T", [1, 33, 500])
def test_f32_items(shape, T):
    wl = workloads.make_workload(small("f32", tokens=T, n_experts=3, **shape))
    assert_parity(wl, *_run(wl))
