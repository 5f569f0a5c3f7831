"""The paths a forward's kernels choose by size, at the sizes where they
switch or leave remainders, against the oracle (rules in gpu_helpers.py)."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_helpers import assert_parity, compare, make_layer, oracle_routing, run_gpu

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


@pytest.mark.parametrize("K,B", [(5, 4), (8, 12), (3, 16), (9, 8), (16, 12), (17, 16), (32, 8),
                                 (33, 4), (6, 32)])
@pytest.mark.parametrize("topk", [0, 2])
def test_decision_instances(K, B, topk):
    """Every instance of the decision step (K up to 8, 16 and 32, B up to 16,
    the general one beyond) with counts that leave entries unused."""
    wl = workloads.make_workload(small(n_experts=K, n_blocks=B, d_ff=64 * B if B != 12 else 768,
                                       topk_fixed=topk))
    assert_parity(wl, *_run(wl))


@pytest.mark.parametrize("K", [8, 16, 32])
def test_decisions_of_tokens_that_are_not_finite(K):
    """A token holding NaN or infinity takes all K residual experts (no prefix
    of its affinities reaches beta) and leaves every other token as it is."""
    s = small(n_experts=K)
    wl = workloads.make_workload(s)
    clean = run_gpu(wl)
    x = wl.x.clone()
    x[7, 3] = float("nan")
    x[100, 0] = float("inf")
    bad = run_gpu(wl, layer=clean.layer, x=x)
    keep = np.ones(s.tokens, bool)
    keep[[7, 100]] = False
    assert (bad.k[~keep] == K).all()
    assert (bad.b[keep] == clean.b[keep]).all() and (bad.k[keep] == clean.k[keep]).all()
    assert (bad.shr[keep] == clean.shr[keep]).all() and (bad.em[keep] == clean.em[keep]).all()


@pytest.mark.parametrize("K", [5, 8, 12, 16, 32])
def test_equal_affinities_go_to_the_lower_expert(K):
    """A zero token's logits are all equal: the first experts are its own."""
    wl = workloads.make_workload(small(n_experts=K, topk_fixed=3))
    x = wl.x.clone()
    x[11] = 0
    g = run_gpu(wl, x=x)
    assert g.k[11] == 3 and int(g.em[11]) == 0b111


@pytest.mark.parametrize("T", [152 * 128, 152 * 128 + 1, 40001])
def test_router_two_ctas_per_sm(T):
    """One wave of 128-token router CTAs, one token more, and a ragged count
    of two waves: decisions, rows and outputs of every token."""
    wl = workloads.make_workload(small(tokens=T, n_experts=2, d_ff=256))
    assert_parity(wl, *_run(wl))


@pytest.mark.parametrize("shape", [
    dict(d_model=72, d_ff=60, n_blocks=4),     # M = 15: unaligned weight columns; d % 32 = 8
    dict(d_model=64, d_ff=280, n_blocks=4),    # M = 70: one whole 64-column item and 6 columns
    dict(d_model=200, d_ff=512, n_blocks=2),   # several reduction steps, d % 64 = 8
])
@pytest.mark.parametrize("T", [1, 33, 500])
def test_f32_items(shape, T):
    wl = workloads.make_workload(small("f32", tokens=T, n_experts=3, **shape))
    assert_parity(wl, *_run(wl))


@pytest.mark.parametrize("shape", [
    dict(d_model=768, d_ff=1536, n_blocks=4),   # two 192-channel sub-tiles
    dict(d_model=832, d_ff=768, n_blocks=4),    # 13 reduction steps, no multiple of the ring
    dict(d_model=1024, d_ff=1024, n_blocks=2),  # 256-channel sub-tiles
    dict(d_model=2048, d_ff=320, n_blocks=5),   # 64-channel blocks
])
@pytest.mark.parametrize("T", [1, 130, 257, 1000])
def test_pair_up_projection(shape, T):
    """Wide layers' up projection on CTA pairs: groups of less than one half
    of a pair tile, of one row into the second half, of several tiles."""
    wl = workloads.make_workload(small(tokens=T, n_experts=2, **shape))
    assert_parity(wl, *_run(wl))


@pytest.mark.parametrize("shape", [
    dict(d_model=832, d_ff=768, n_blocks=4, n_experts=2),    # one bundle
    dict(d_model=1024, d_ff=1024, n_blocks=8, n_experts=1),  # two
    dict(d_model=768, d_ff=3072, n_blocks=16, n_experts=2),  # four
])
@pytest.mark.parametrize("kw", [dict(), dict(topk_fixed=1), dict(prefix_blocks=1),
                                dict(alpha_fixed=0.0), dict(seq_len=100, min_len=1)])
def test_bundled_down_projection(shape, kw):
    """Passes of enough tokens for the down projection's rows to be bundled
    over four blocks: every pattern, only full ones (alpha = 0: no shared
    block, all blocks of every residual expert), prefixes, padding."""
    wl = workloads.make_workload(small(tokens=5111, **shape, **kw))
    g, rep = _run(wl)
    assert g.layer.kernels_per_forward() == 6
    assert_parity(wl, g, rep)
    # a smaller forward on the same handle takes the unbundled kernels, and
    # the next large one the bundled ones again
    few = run_gpu(wl, layer=g.layer, x=wl.x[:200].clone(),
                  mask=None if wl.mask is None else wl.mask[:200])
    assert (few.b == g.b[:200]).all() and (few.k == g.k[:200]).all()
    again = run_gpu(wl, layer=g.layer)
    # (h is rounded to bf16 alike: the fp32 sums' order and one rounding to bf16)
    for y, ref in ((few.y, g.y[:200]), (again.y, g.y)):
        assert (np.abs(y - ref).max(axis=1) <= 2.0 ** -7 * np.abs(ref).max(axis=1)).all()


@pytest.mark.parametrize("T,kw,kernels", [
    (3000, dict(), 6), (3000, dict(beta_fixed=0.05), 4), (3000, dict(alpha_fixed=0.95), 4),
    (6000, dict(beta_fixed=0.05), 6), (3000, dict(beta_fixed=0.9), 6),
])
def test_few_experts_per_token_bundle_later(T, kw, kernels):
    """A fixed mass that one expert reaches leaves fewer rows per group: the
    bundled down projection begins at more tokens."""
    wl = workloads.make_workload(small(tokens=T, d_model=832, d_ff=768, n_experts=9, **kw))
    g, rep = _run(wl)
    assert g.layer.kernels_per_forward() == kernels
    assert_parity(wl, g, rep)


@pytest.mark.parametrize("T,d,masked", [(14335, 256, False), (14336, 256, True),
                                        (20011, 256, False), (28671, 128, True),
                                        (28672, 128, False)])
def test_host_forward_in_parts(T, d, masked):
    """From 14,336 tokens and 7 MiB on, a forward of pinned buffers runs in three
    parts: outputs, counts, records and the group table as of one pass."""
    s = small(tokens=T, d_model=d, n_experts=2, d_ff=256,
              **(dict(seq_len=50, min_len=1) if masked else {}))
    wl = workloads.make_workload(s)
    g = run_gpu(wl)
    counts, offsets, tok, w = g.layer.groups()
    out = torch.empty_like(wl.x).pin_memory()
    b = torch.empty(T, dtype=torch.int32).pin_memory()
    k = torch.empty(T, dtype=torch.int32).pin_memory()
    mask = None if wl.mask is None else wl.mask.pin_memory()
    for _ in range(2):  # both accumulators
        out.fill_(7.0)
        g.layer.forward_host(wl.x.pin_memory(), out, mask, b, k)
        assert g.layer.sync_status() == 0
        assert (b.numpy() == g.b).all() and (k.numpy() == g.k).all()
        y = out.float().numpy()
        assert np.abs(y - g.y).max() <= 2.0 ** -7 * np.abs(g.y).max()
    again = g.layer.groups()
    assert torch.equal(again[0], counts) and torch.equal(again[2], tok)
    assert torch.equal(again[3], w)


@pytest.mark.parametrize("shift", [0, 15000, -10000, 3])
def test_host_forward_of_overlapping_buffers(shift):
    """x and out in one pinned buffer, out `shift` rows after x: as with buffers
    of their own (x is read before any of it is overwritten)."""
    T, d = 20000, 384
    wl = workloads.make_workload(small(tokens=T, d_model=d, n_experts=2))
    g = run_gpu(wl)
    for _ in range(3):
        buf = torch.zeros(T + abs(shift), d, dtype=torch.bfloat16).pin_memory()
        x, out = buf[max(-shift, 0):][:T], buf[max(shift, 0):][:T]
        x.copy_(wl.x)
        g.layer.forward_host(x, out)
        assert g.layer.sync_status() == 0
        assert np.abs(out.float().numpy() - g.y).max() <= 2.0 ** -7 * np.abs(g.y).max()


@pytest.mark.parametrize("kw", [
    dict(tokens=3000, n_experts=2),                   # groups of more than one chunk: added
    dict(tokens=900, n_experts=3, d_ff=768),          # single chunks: stored (M = 192)
    dict(tokens=900, n_experts=3, alpha_fixed=1.0),   # empty groups: cleared
    dict(tokens=1100, n_experts=2, d_model=768, d_ff=1536),  # two N chunks, six feature chunks
    dict(tokens=4200, n_experts=2),                   # dL/dx by the weight-stationary kernel
    dict(tokens=4200, n_experts=1, d_model=768, d_ff=768),  # the same in column slices
])
def test_weight_gradient_chunks(kw):
    """Weight gradients of groups that are one chunk, several, or empty, the
    buffers filled with NaN before: every entry is written."""
    from test_gpu_backward import check, run_case
    wl, got, ref, L = run_case(small(**kw))
    check(wl, got, ref)
    dev = torch.device("cuda")
    x, dy = wl.x.to(dev), torch.ones_like(wl.x, device=dev)
    a = L.backward(x, dy, want_bias=True)
    # the same into buffers on 16-byte, not 32-byte boundaries
    def odd(t):
        flat = torch.full((t.numel() + 4,), float("nan"), device=dev)
        return flat[4:].view(t.shape)
    b = L.backward(x, dy, want_bias=True, out={k: odd(v) for k, v in a.items()})
    torch.cuda.synchronize()
    for k in ("dx", "dw_up", "dw_down", "dw_router", "dbias"):
        assert torch.isfinite(b[k]).all(), k
        # (two runs: fp32 sums in another order, of up to 3,000 terms)
        assert (a[k] - b[k]).abs().max() <= 1e-4 * a[k].abs().max(), k


@pytest.mark.parametrize("shape", [
    dict(d_model=128, d_ff=512, n_blocks=4),   # both projections weight-stationary
    # the down projection alone, in column slices (no whole bundles of four blocks)
    dict(d_model=768, d_ff=1152, n_blocks=6),
    dict(d_model=256, d_ff=1536, n_blocks=4),  # two sub-tiles per block: the up projection streams
])
@pytest.mark.parametrize("T", [4095, 4096, 4321])
def test_grouped_kernels_around_the_weight_stationary_switch(shape, T):
    """Below 4,096 tokens grouped layers run the pair and streaming kernels,
    from there on the weight-stationary ones where they fit."""
    wl = workloads.make_workload(small(tokens=T, n_experts=2, topk_fixed=1, **shape))
    g = run_gpu(wl, gemm_kernels="grouped")
    assert g.layer.kernels_per_forward() == 4
    assert_parity(wl, g, compare(wl, g))


@pytest.mark.parametrize("K,B,T,kw", [
    (16, 12, 1, dict()),                         # one token
    (8, 16, 5003, dict()),                       # two chunks per CTA, a ragged last one
    (15, 8, 12001, dict(topk_fixed=1)),          # three; 128 groups
    (7, 20, 700, dict()),                        # more blocks than the unrolled loop takes
    (2, 64, 300, dict(seq_len=100, min_len=1)),  # whole block masks, padding
    (16, 16, 700, dict(alpha_fixed=0.0, topk_fixed=16)),  # more rows than fit: one by one
])
def test_router_rows_staged(K, B, T, kw):
    """Group rows put together in shared memory (from 128 groups on): outputs,
    and the group table against the decisions."""
    wl = workloads.make_workload(small(tokens=T, d_ff=64 * B, n_experts=K, n_blocks=B, **kw))
    g = run_gpu(wl, gemm_kernels="grouped")
    assert_parity(wl, g, compare(wl, g))
    counts, offsets, tok, w = (v.numpy() for v in g.layer.groups())
    r = oracle.with_decisions(oracle_routing(wl), g.shr, g.em, B)
    c_ref, tok_ref, w_ref = oracle.groups(r, K, B, *([] if wl.mask is None else [wl.mask.numpy()]))
    assert counts.tolist() == c_ref.tolist()
    real = tok >= 0
    assert tok[real].tolist() == tok_ref.tolist()
    np.testing.assert_allclose(w[real], w_ref, rtol=1e-5, atol=1e-7)
