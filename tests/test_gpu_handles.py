"""Handles of different shapes in one process, and handles that find little
memory left."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def make(d, H, K, B, T, dtype="bf16", train=False, max_tokens=None, **kw):
    """A layer with random weights, its tokens and its output gradient."""
    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT, Layer
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(7)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16

    def randn(*shape, scale=1.0):
        return (torch.randn(*shape, generator=g, device=dev) * scale).to(dt)

    layer = Layer(d, H, K, B, dtype=dtype, max_tokens=max_tokens or T,
                  features=FEATURES_DEFAULT | (FEATURE_BACKWARD if train else 0), **kw)
    layer.load_weights(randn(d, K + 1, scale=0.02), randn(K + 1, H, d, scale=d ** -0.5),
                       randn(K + 1, d, H, scale=H ** -0.5))
    return layer, randn(T, d), randn(T, d, scale=0.01)


def outputs(layer, x, dy, train):
    out = [layer.forward(x).float()]
    if train:
        g = layer.backward(x, dy, want_bias=True)
        out += [g[k] for k in ("dx", "dw_up", "dw_down", "dw_router", "dbias")]
    torch.cuda.synchronize()
    assert layer.sync_status() == 0
    return out


@pytest.mark.parametrize("large,small,kernels", [
    # (kernels per forward of `large`: the path meant)
    (dict(d=768, H=3072, K=16, B=8, T=300), dict(d=768, H=3072, K=8, B=8, T=300), 4),  # CTA pairs
    (dict(d=640, H=3072, K=32, B=16, T=3500), dict(d=640, H=3072, K=16, B=16, T=3500), 6),  # bundles
    (dict(d=384, H=1536, K=16, B=8, T=300, max_tokens=80000),
     dict(d=384, H=1536, K=8, B=8, T=300), 3),  # expert tiles
    (dict(d=384, H=1536, K=16, B=8, T=4200, gemm_kernels="grouped"),
     dict(d=384, H=1536, K=4, B=8, T=4200, gemm_kernels="grouped"), 4),  # weight-stationary
    (dict(d=768, H=3072, K=16, B=16, T=500, train=True),
     dict(d=768, H=3072, K=8, B=8, T=500, train=True), 4),
    (dict(d=64, H=256, K=32, B=16, T=200, dtype="f32"),
     dict(d=64, H=256, K=4, B=4, T=200, dtype="f32"), 6),
])
def test_a_later_handle_leaves_an_earlier_one_as_it_is(large, small, kernels):
    """A handle whose kernels need less shared memory than those of a handle
    made before it: both run, the first one with the outputs it had (up to the
    order of fp32 sums into the output, then one rounding to bf16)."""
    train = large.get("train", False)
    a, x, dy = make(**large)
    assert a.kernels_per_forward() == kernels
    before = outputs(a, x, dy, train)
    b, xb, dyb = make(**small)
    after = outputs(a, x, dy, train)
    outputs(b, xb, dyb, train)
    for u, v in zip(before, after):
        assert (u - v).abs().max() <= 2.0 ** -7 * u.abs().max()


def test_a_handle_without_room_for_the_bundles_is_made_unbundled():
    """With too little memory left for the bundled down projection's tables, but
    enough for everything else of a training handle, the handle is made and runs
    the unbundled kernels."""
    from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT, Layer
    T, shape = 16000, (640, 3072, 32, 16)

    def layer():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        made = Layer(*shape, max_tokens=T, features=FEATURES_DEFAULT | FEATURE_BACKWARD)
        return made, free - torch.cuda.mem_get_info()[0]

    src, x, dy = make(*shape, T)
    weights = src._keep[:3]
    del src
    a, size = layer()
    assert a.kernels_per_forward() == 6
    a.load_weights(*weights)
    y = a.forward(x).float()
    grads = a.backward(x, dy)
    a.close()
    # the tables and the larger h take 0.4 GB: leave all but half of that
    room = size - (200 << 20)
    held = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    b, smaller = layer()
    try:
        assert b.kernels_per_forward() == 4 and smaller < room
        b.load_weights(*weights)
        out = b.forward(x)
        b.backward(x, dy, out=grads)
        torch.cuda.synchronize()
        assert b.sync_status() == 0
    finally:
        b.close()
        del held
        torch.cuda.empty_cache()
    assert (out.float() - y).abs().max() <= 2.0 ** -7 * y.abs().max()
