"""Backward pass on the GPU (training, Sec. III-E) against the oracle.

The gradients are defined with the forward's discrete decisions held fixed,
so the oracle's backward runs on the GPU's own decisions (their parity with
the oracle's is the forward tests' subject); alpha and s are the oracle's,
recomputed in fp64 from the same bf16 inputs and weights.

Tolerance: the GPU keeps dL/da and w GeLU(a) in bf16 (8 significant bits,
2^-8 relative) between its GEMMs and accumulates in fp32, as the forward
keeps h; every gradient is compared at the forward's bf16 bound of 2e-2:
dL/dx per token (max |err| / max |ref| over the token's features), each
weight gradient over the whole tensor (max |err| / max |ref|)."""
import math

import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_helpers import make_layer, thresholds_of

pytestmark = pytest.mark.gpu

TOL = 2e-2


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def run_case(spec, lambda_div=0.0, seed=11):
    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT
    wl = workloads.make_workload(spec)
    dev = torch.device("cuda")
    L = make_layer(spec, features=FEATURES_DEFAULT | FEATURE_BACKWARD)
    bias = None if wl.router_bias is None else wl.router_bias.to(dev)
    L.load_weights(wl.w_router.to(dev), wl.w_up.to(dev), wl.w_down.to(dev), bias)
    x = wl.x.to(dev)
    md = None if wl.mask is None else wl.mask.to(dev)
    L.forward(x, mask=md)
    r = L.routing()
    g = torch.Generator().manual_seed(seed)
    dy = torch.randn(spec.tokens, spec.d_model, generator=g).to(torch.bfloat16)
    grads = L.backward(x, dy.to(dev), mask=md, lambda_div=lambda_div, want_bias=True)
    torch.cuda.synchronize()
    assert L.sync_status() == 0
    got = {k: (None if v is None else v.double().cpu().numpy()) for k, v in grads.items()}
    shr = r["shared_mask"].cpu().numpy().view(np.uint64)
    em = r["expert_mask"].cpu().numpy().view(np.uint64)
    ref = oracle.backward(wl.x, wl.w_router, wl.w_up, wl.w_down, shr, em, spec.n_blocks, dy,
                          thresholds_of(spec), wl.mask, wl.router_bias)
    return wl, got, ref, L


def rel_tensor(got, ref):
    return float(np.abs(got - ref).max() / max(np.abs(ref).max(), 1e-30))


def rel_rows(got, ref, valid):
    den = np.abs(ref).max(axis=1)
    err = np.abs(got - ref).max(axis=1)
    ok = valid & (den > 0)
    return float((err[ok] / den[ok]).max()) if ok.any() else 0.0


def check(wl, got, ref, lambda_div=0.0):
    T = wl.x.shape[0]
    valid = np.ones(T, bool) if wl.mask is None else wl.mask.numpy() != 0
    assert np.isfinite(got["dx"]).all()
    assert (got["dx"][~valid] == 0).all()
    errs = {"dx": rel_rows(got["dx"], ref.dx, valid),
            "dw_up": rel_tensor(got["dw_up"], ref.dw_up),
            "dw_down": rel_tensor(got["dw_down"], ref.dw_down),
            "dbias": rel_tensor(got["dbias"], ref.dbias)}
    wr_ref = ref.dw_router
    if lambda_div:
        _, gdiv = oracle.diversity(wl.w_router)
        wr_ref = wr_ref + lambda_div * gdiv
    errs["dw_router"] = rel_tensor(got["dw_router"], wr_ref)
    print(errs)
    for k, v in errs.items():
        assert v <= TOL, (k, v, errs)
    return errs


def small(**kw):
    base = dict(tokens=300, d_model=128, d_ff=512, n_experts=4, n_blocks=4)
    base.update(kw)
    return workloads.spec("vit_s").with_(**base)


def test_backward_small_ragged():
    """300 tokens: the last tile of every group is ragged."""
    wl, got, ref, _ = run_case(small())
    check(wl, got, ref)


def test_backward_vit_s_full_size():
    wl, got, ref, _ = run_case(workloads.spec("vit_s"))
    check(wl, got, ref)


def test_backward_bert_padding_two_subtiles():
    """BERT-base: block width 384 runs as two 192-channel sub-tiles in both
    backward GEMM kernels; padding tokens (NaN inputs) get dx = 0."""
    wl, got, ref, _ = run_case(workloads.spec("bert_base"))
    check(wl, got, ref)


def test_backward_router_bias_many_experts():
    """The stress layer's shapes (K = 32, B = 16, d = 1024) and Zipf router
    bias on its first 2,048 tokens: the bias gradient and 33 router columns."""
    wl, got, ref, _ = run_case(workloads.spec("stress", tokens=2048))
    check(wl, got, ref)


def test_backward_sixteen_experts():
    """K = 16 residual experts (17 router columns, as ViT-B's layer), 300
    tokens: the router gradients' kernel instance for up to 32 columns."""
    wl, got, ref, _ = run_case(small(tokens=300, n_experts=16))
    check(wl, got, ref)


def test_backward_gram_regulariser():
    """lambda_div = 0.01 (the paper's choice): dW* gains lambda dL_div/dW*,
    and L_div itself is returned."""
    lam = 0.01
    wl, got, ref, _ = run_case(small(tokens=500), lambda_div=lam)
    check(wl, got, ref, lambda_div=lam)
    L, _ = oracle.diversity(wl.w_router)
    assert got["l_div"][0] == pytest.approx(L, rel=1e-4)


def test_backward_fixed_alpha_has_no_shared_router_gradient():
    wl, got, ref, _ = run_case(small(tokens=400, alpha_fixed=0.4))
    check(wl, got, ref)
    assert (got["dw_router"][:, 0] == 0).all()


def test_backward_argument_errors():
    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT, UnifMoeError
    s = small(tokens=256)
    wl = workloads.make_workload(s)
    dev = torch.device("cuda")
    x = wl.x.to(dev)
    dy = torch.zeros_like(x)
    plain = make_layer(s)
    plain.load_weights(wl.w_router.to(dev), wl.w_up.to(dev), wl.w_down.to(dev))
    plain.forward(x)
    with pytest.raises(UnifMoeError) as e:  # no backward workspace
        plain.backward(x, dy)
    assert e.value.code == -6
    L = make_layer(s, features=FEATURES_DEFAULT | FEATURE_BACKWARD)
    L.load_weights(wl.w_router.to(dev), wl.w_up.to(dev), wl.w_down.to(dev))
    with pytest.raises(UnifMoeError) as e:  # no forward yet
        L.backward(x, dy)
    assert e.value.code == -6
    L.forward(x)
    with pytest.raises(UnifMoeError) as e:  # another T than the forward's
        L.backward(x[:100], dy[:100])
    assert e.value.code == -6
    torch.cuda.synchronize()
    assert L.sync_status() == 0


def test_gelu_of_the_router_gradient_in_fp32():
    """dL/dalpha takes GeLU(a) in fp32. Token t has x = a_t in feature 0, whose
    key is 1 in the shared expert's first channel, and 1 in feature 1 + t; dy V^T
    is 1 in that channel; alpha = 1/2 (zero router, tau = 0, one of two blocks
    shared): dL/dW*[1 + t][0] = GeLU(a_t) / 4, all other factors and terms being
    exact. For every bf16 a_t of [2^-6, 8) and both signs.

    Bound: Phi's sum is rounded by 2^-25. For |a| < 1.35, P by 2^-26 (times |a|) and
    less before it, 7e-8 in all. Beyond, Phi(-|a|) <= 0.089 times the errors of the
    exponential (2^-22 and its argument's), the reciprocal (2^-23) and three
    roundings, 8.5e-8 in all. Below 2^-23 |a|, then; the product's rounding adds
    2^-24 |GeLU|. (erff within its documented 2 ulp gives the same bound.)"""
    from scipy.stats import norm

    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT, Layer
    dev, d, H, T = torch.device("cuda"), 1024, 128, 1000
    L = Layer(d, H, 1, 2, max_tokens=T, tau=0.0, prefix_blocks=1,
              features=FEATURES_DEFAULT | FEATURE_BACKWARD)
    zeros = dict(dtype=torch.bfloat16, device=dev)
    w_up, w_down = torch.zeros(2, H, d, **zeros), torch.zeros(2, d, H, **zeros)
    w_up[0, 0, 0] = w_down[0, 0, 0] = 1
    L.load_weights(torch.zeros(d, 2, **zeros), w_up, w_down)
    mag = (torch.arange(128, dtype=torch.float64) / 128 + 1) * 2.0 ** torch.arange(
        -6, 3, dtype=torch.float64)[:, None]
    values = torch.cat([mag.flatten(), -mag.flatten()])
    dy = torch.zeros(T, d, **zeros)
    dy[:, 0] = 1
    worst = 0.0
    for a in values.split(T):
        x = torch.zeros(T, d, **zeros)
        x[:a.numel(), 0] = a.to(dev, torch.bfloat16)
        x[torch.arange(T), 1 + torch.arange(T)] = 1
        L.forward(x)
        dw = L.backward(x, dy)["dw_router"]
        torch.cuda.synchronize()
        assert L.sync_status() == 0
        got = 4 * dw[1:1 + a.numel(), 0].double().cpu().numpy()
        ref = a.numpy() * norm.cdf(a.numpy())
        bound = 2.0 ** -23 * np.abs(a.numpy()) + 2.0 ** -24 * np.abs(ref)
        worst = max(worst, float((np.abs(got - ref) / bound).max()))
    assert worst <= 1.0, worst


@pytest.mark.parametrize("T,alpha,topk,shape", [
    # 57 groups of 99 tiles, one item per group: 13 sums, stored and added
    (12608, 0.125, 8, dict(d_model=384, d_ff=1536, n_experts=8, n_blocks=8)),
    # 9 tiles per group
    (1025, 0.125, 8, dict(d_model=384, d_ff=1536, n_experts=8, n_blocks=8)),
    # 3 groups of 313 tiles, 13 items per group, 4 sums each
    (40003, 0.5, 2, dict(d_model=512, d_ff=256, n_experts=2, n_blocks=2)),
])
def test_weight_gradient_accumulation_error(T, alpha, topk, shape):
    """dV over groups of T rows, all rows of w GeLU(a) being equal (the same x for
    every token): dV[i][h] = (sum_t dy[t][i]) hw[h], with hw an exact bf16 number
    that the results give themselves. dy > 0, so that nothing cancels.

    Bound: 1,024 rows are 64 accumulations, each truncated below the last bit
    of the sum (2^-23 of it, half of that on average over a growing sum), then
    at most T / 1,024 fp32 additions of 2^-24 each."""
    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT
    s = small(tokens=T, alpha_fixed=alpha, topk_fixed=topk, **shape)
    wl = workloads.make_workload(s)
    dev = torch.device("cuda")
    L = make_layer(s, features=FEATURES_DEFAULT | FEATURE_BACKWARD)
    L.load_weights(wl.w_router.to(dev), wl.w_up.to(dev), wl.w_down.to(dev))
    x = wl.x[:1].to(dev).expand(T, -1).contiguous()
    g = torch.Generator().manual_seed(3)
    dy = torch.rand(T, s.d_model, generator=g).to(torch.bfloat16).to(dev)
    L.forward(x)
    dv = L.backward(x, dy)["dw_down"].double()
    torch.cuda.synchronize()
    assert L.sync_status() == 0
    total = dy.double().sum(0)
    hw = (dv / total[None, :, None]).mean(1).to(torch.bfloat16).double()  # [K + 1][H]
    assert (hw != 0).any(dim=1).sum() == 1 + topk  # the experts that run
    ref = total[None, :, None] * hw[:, None, :]
    err = ((dv - ref).abs() / ref.abs())[ref != 0].max()
    assert (dv[ref == 0] == 0).all()
    assert err <= 64 * 2.0 ** -24 + T / 1024 * 2.0 ** -24, float(err)
