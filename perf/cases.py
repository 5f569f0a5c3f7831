"""The work that programs have this framework do, as cases to be measured.

A case is one UniF-MoE layer (d features, FFN width H, K residual experts, B
blocks, a dtype), a number of token slots T, the options in use and the entry
point called: "forward" (the layer alone, as in an inference engine),
"sublayer" (the layer inside its Transformer sublayer), "train" (forward, then
backward with the Gram regulariser) or "host" (a forward of host buffers).
Shapes are those of the workloads package (DeiT-S, BERT-base and ViT-B FFNs, a
1,024-wide load-imbalanced layer, a small fp32 layer) with the paper's range of
experts and blocks (K = 6..16, B = 8..16; 32 for the wide layer); inputs follow
the same distributions, drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2608_10392_gb300 import FEATURE_BACKWARD, FEATURES_DEFAULT, Layer

ADAPTIVE = dict(alpha_fixed=-1.0, beta_fixed=-1.0, topk=0, prefix=False)


def _case(name, call, T, d, H, K, B, dtype="bf16", seq=0, skew=False, norm_first=False, **options):
    c = dict(name=name, call=call, T=T, d=d, H=H, K=K, B=B, dtype=dtype, seq=seq, skew=skew,
             norm_first=norm_first, **ADAPTIVE)
    c.update(options)
    return c


def listed():
    return [
        # one 197-token image through the layer: online inference, where latency counts
        _case("vit_s_image", "forward", 197, 384, 1536, 8, 8),
        # eight images through a whole pre-norm sublayer, as DeiT-S holds the layer
        _case("vit_s_sublayer", "sublayer", 8 * 197, 384, 1536, 8, 8, norm_first=True),
        # an odd number of tokens, two residual experts per token (the fixed-count ablation)
        _case("vit_s_top2", "forward", 5003, 384, 1536, 8, 8, topk=2),
        # the evaluation batch of 64 images
        _case("vit_s_batch", "forward", 64 * 197, 384, 1536, 8, 8),
        # the same from pinned host buffers, copies included
        _case("vit_s_host", "host", 64 * 197, 384, 1536, 8, 8),
        # a training step on that batch: forward, backward, Gram regulariser
        _case("vit_s_train", "train", 64 * 197, 384, 1536, 8, 8),
        # one 128-token sentence
        _case("bert_sentence", "forward", 128, 768, 3072, 8, 8, seq=128),
        # 32 padded sentences through a whole post-norm sublayer, as BERT holds the layer
        _case("bert_sublayer", "sublayer", 32 * 128, 768, 3072, 8, 8, seq=128),
        # a training step on 32 padded sentences
        _case("bert_train", "train", 32 * 128, 768, 3072, 8, 8, seq=128),
        # the evaluation batch through the wider layer with twice the experts and blocks
        _case("vit_b_batch", "forward", 64 * 197, 768, 3072, 16, 16),
        # throughput serving of many tokens with unevenly popular experts
        _case("wide_skewed", "forward", 65536, 1024, 4096, 32, 16, skew=True),
        # the small fp32 layer
        _case("small_f32", "forward", 256, 64, 256, 4, 4, dtype="f32"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["forward", "forward", "forward", "sublayer", "sublayer", "train", "train",
                       "host"])
    family = rng.choice(["s", "s", "b", "b", "wide", "f32"]) if call in ("forward", "sublayer") \
        else rng.choice(["s", "b"])
    seq, skew, dtype = 0, False, "bf16"
    if family == "s":
        d, H, B, K = 384, 1536, rng.choice([8, 12]), rng.randint(6, 16)
        T = _spread(rng, 100, 40000)
    elif family == "b":
        d, H, B, K = 768, 3072, rng.choice([8, 12, 16]), rng.randint(6, 16)
        T = _spread(rng, 100, 16000)
    elif family == "wide":
        d, H, B, K, skew = 1024, 4096, rng.choice([8, 16]), rng.randint(8, 32), True
        T = _spread(rng, 1000, 40000)
    else:
        d, H, B, K, dtype = 64, 256, 4, rng.randint(2, 8), "f32"
        T = _spread(rng, 50, 2000)
    if call == "train":
        T = min(T, 16000 if family == "s" else 6000)
    if family in ("s", "b") and rng.random() < 0.4:  # padded sequences of one length
        seq = rng.choice([64, 128, 197])
    options = dict(ADAPTIVE)
    if family != "f32":
        options.update(rng.choice([{}, {}, {}, dict(topk=2), dict(alpha_fixed=0.4),
                                   dict(beta_fixed=0.7), dict(prefix=True)]))
    c = _case("", call, T, d, H, K, B, dtype=dtype, seq=seq, skew=skew,
              norm_first=rng.random() < 0.5, **options)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _inputs(case, seed, device):
    """Weights (experts: one base FFN plus 5% noise; router columns N(0, 0.02)),
    tokens N(0, 1) (layer-normalised activations; for a skewed layer a mixture
    that spans the shared score and favours four experts, with a Zipf router
    bias), the padding mask with NaN in the padded rows, the gradient of the
    output for a training step, and the sublayer's norm parameters."""
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 7919 + 13)
    f = dict(generator=g, device=device, dtype=torch.float32)
    T, d, H, K = case["T"], case["d"], case["H"], case["K"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    s1, s2 = 1.0 / math.sqrt(d), 1.0 / math.sqrt(H)
    base_up, base_down = torch.randn(H, d, **f) * s1, torch.randn(d, H, **f) * s2
    w_up = torch.empty(K + 1, H, d, device=device, dtype=dt)
    w_down = torch.empty(K + 1, d, H, device=device, dtype=dt)
    for e in range(K + 1):
        w_up[e] = base_up + torch.randn(H, d, **f) * (0.05 * s1)
        w_down[e] = base_down + torch.randn(d, H, **f) * (0.05 * s2)
    w_router = (torch.randn(d, K + 1, **f) * 0.02).to(dt)
    bias = None
    x = torch.randn(T, d, **f)
    if case["skew"]:
        bias = torch.zeros(K + 1, device=device)
        bias[1:] = -1.2 * torch.log(torch.arange(1, K + 1, device=device, dtype=torch.float32))
        wr = w_router.float()
        means = torch.stack([
            shift / wr[:, 0].norm() ** 2 * wr[:, 0]
            + 4.0 / wr[:, 1 + c * (K // 4)].norm() ** 2 * wr[:, 1 + c * (K // 4)]
            for c, shift in enumerate((-8.0, -2.0, 2.0, 8.0))])
        x += means[torch.randint(0, 4, (T,), generator=g, device=device)]
    mask = None
    if case["seq"]:
        n = (T + case["seq"] - 1) // case["seq"]
        lens = torch.randint(case["seq"] // 8, case["seq"] + 1, (n,), generator=g, device=device)
        mask = (torch.arange(case["seq"], device=device) < lens[:, None]).reshape(-1)[:T]
        x[~mask] = float("nan")
        mask = mask.to(torch.uint8)
    v = dict(w_router=w_router, w_up=w_up, w_down=w_down, bias=bias, x=x.to(dt), mask=mask)
    if case["call"] == "train":
        v["dy"] = (torch.randn(T, d, **f) * 0.01).to(dt)
    if case["call"] == "sublayer":
        v["gamma"] = (1 + 0.1 * torch.randn(d, **f)).to(dt)
        v["beta"] = (0.1 * torch.randn(d, **f)).to(dt)
    return v


LAMBDA_DIV, EPS = 0.01, 1e-6


def prepare(case, seed):
    v = _inputs(case, seed, torch.device("cuda"))
    layer = Layer(case["d"], case["H"], case["K"], case["B"], dtype=case["dtype"],
                  max_tokens=case["T"],
                  alpha_fixed=case["alpha_fixed"] if case["alpha_fixed"] >= 0 else math.nan,
                  beta_fixed=case["beta_fixed"] if case["beta_fixed"] >= 0 else math.nan,
                  topk_fixed=case["topk"], prefix_blocks=int(case["prefix"]),
                  features=FEATURES_DEFAULT | (FEATURE_BACKWARD if case["call"] == "train" else 0))
    layer.load_weights(v["w_router"], v["w_up"], v["w_down"], v["bias"])
    T = case["T"]
    s = dict(case=case, layer=layer, x=v["x"], mask=v["mask"], gamma=v.get("gamma"),
             beta=v.get("beta"), dy=v.get("dy"), grads=None)
    if case["call"] == "host":
        for k in ("x", "mask"):
            s[k] = None if s[k] is None else s[k].cpu().pin_memory()
        s["out"] = torch.empty_like(s["x"]).pin_memory()
        s["b"] = torch.empty(T, dtype=torch.int32).pin_memory()
        s["k"] = torch.empty(T, dtype=torch.int32).pin_memory()
    else:
        s["b"] = torch.empty(T, dtype=torch.int32, device="cuda")
        s["k"] = torch.empty(T, dtype=torch.int32, device="cuda")
    return s


def run(s):
    case, layer = s["case"], s["layer"]
    if case["call"] == "host":
        layer.forward_host(s["x"], s["out"], s["mask"], s["b"], s["k"])
        return dict(y=s["out"], b=s["b"], k=s["k"])
    if case["call"] == "sublayer":
        y = layer.sublayer_forward(s["x"], s["gamma"], s["beta"], EPS, case["norm_first"],
                                   mask=s["mask"], shared_counts=s["b"], residual_counts=s["k"])
        return dict(y=y, b=s["b"], k=s["k"])
    y = layer.forward(s["x"], mask=s["mask"], shared_counts=s["b"], residual_counts=s["k"])
    if case["call"] == "forward":
        return dict(y=y, b=s["b"], k=s["k"])
    # the gradient buffers are the program's own, filled again in every step
    s["grads"] = layer.backward(s["x"], s["dy"], mask=s["mask"], lambda_div=LAMBDA_DIV,
                                want_bias=True, out=s["grads"])
    return dict(y=y, b=s["b"], k=s["k"], **s["grads"])


# ------------------------------------------------------------------ work

def _mean_blocks(case):
    """Mean C_B = b + k (B - b) per valid token over the case's distribution of
    router logits (column norm 0.02 sqrt(d), tokens N(0, 1))."""
    r = np.random.RandomState(3)
    n, K, B = 4000, case["K"], case["B"]
    sd = 0.02 * math.sqrt(case["d"])
    z = r.randn(n, K + 1) * sd
    if case["skew"]:
        c = r.randint(0, 4, n)
        z[:, 0] += np.array([-8.0, -2.0, 2.0, 8.0])[c]
        z[:, 1:] -= 1.2 * np.log(np.arange(1, K + 1))
        z[np.arange(n), 1 + c * (K // 4)] += 4.0
    tau = (B - 1) / B ** 2
    alpha = tau + (1 - 2 * tau) / (1 + np.exp(-z[:, 0]))
    if case["alpha_fixed"] >= 0:
        alpha[:] = case["alpha_fixed"]
    b = np.rint(B * alpha)
    s = np.exp(z[:, 1:])
    s = -np.sort(-s / s.sum(1, keepdims=True), axis=1)
    need = case["beta_fixed"] if case["beta_fixed"] >= 0 else 1 - alpha[:, None]
    k = np.minimum(K, 1 + (np.cumsum(s, axis=1) < need).sum(1))
    if case["topk"]:
        k[:] = case["topk"]
    return float((b + k * (B - b)).mean())


def work(case):
    T, d, H, K, B = (case[k] for k in ("T", "d", "H", "K", "B"))
    es = 4 if case["dtype"] == "f32" else 2
    valid = T * 0.56 if case["seq"] else T
    weights = 2 * (K + 1) * H * d * es + (K + 1 + B) * d * es
    flops = 4 * d * (H // B) * _mean_blocks(case) * valid + 2 * d * (K + 1 + B) * valid
    nbytes = weights + 2 * T * d * es + 8 * T
    if case["call"] == "train":
        flops += 10 * d * (H // B) * _mean_blocks(case) * valid + 4 * d * (K + 1) * valid
        nbytes += weights + 2 * T * d * es + 4 * T * d + 4 * (2 * (K + 1) * H * d + d * (K + 1))
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    # bf16: h and the output are rounded to 8 bits (about 2e-3 against 64 bits), dL/da and the
    # weighted h of a training step too; fp32 sums in another order otherwise. A token whose
    # decision is a near-tie may take another count. Seen against exact(): 2.6e-3 at most for
    # bf16, 2e-7 for fp32.
    if case["dtype"] == "f32":
        return dict(rel=1e-6, differ=0.002)
    return dict(rel=1e-2, differ=0.002)


# ------------------------------------------------------------------ exact

def _gelu(a):
    return 0.5 * a * (1 + torch.erf(a / math.sqrt(2.0)))


def _layernorm(v, gamma, beta):
    c = v - v.mean(1, keepdim=True)
    return gamma * c / torch.sqrt((c * c).mean(1, keepdim=True) + EPS) + beta


def _route(case, v, x):
    """Eqs. 17-27 in 64 bits: alpha, affinities s, the shared block set and the
    selected residual experts of every token, and the shared logit's sigmoid."""
    K, B = case["K"], case["B"]
    tau = (B - 1) / B ** 2
    z = x @ v["w_router"].double()
    if v["bias"] is not None:
        z = z + v["bias"].double()
    sg = torch.sigmoid(z[:, 0])
    alpha = tau + (1 - 2 * tau) * sg
    if case["alpha_fixed"] >= 0:
        alpha = torch.full_like(alpha, float(np.float32(case["alpha_fixed"])))
    b = torch.round(B * alpha).long()
    # block prototypes: the mean of the shared keys, rounded once to the layer dtype
    mu = v["w_up"][0].double().reshape(B, -1, case["d"]).mean(1).to(v["w_up"].dtype).double()
    if case["prefix"]:
        rank = torch.arange(B, device=x.device).expand(x.shape[0], B)
    else:
        order = torch.sort(x @ mu.T, dim=1, descending=True, stable=True)[1]
        rank = torch.empty_like(order).scatter_(
            1, order, torch.arange(B, device=x.device).expand_as(order).contiguous())
    shared = rank < b[:, None]
    s = torch.softmax(z[:, 1:], dim=1)
    p, q = torch.sort(s, dim=1, descending=True, stable=True)
    need = float(np.float32(case["beta_fixed"])) if case["beta_fixed"] >= 0 else 1 - alpha[:, None]
    k = torch.clamp(1 + (torch.cumsum(p, dim=1) < need).sum(1), max=K)
    if case["topk"]:
        k = torch.full_like(k, case["topk"])
    chosen = torch.zeros(x.shape[0], K, dtype=torch.bool, device=x.device).scatter_(
        1, q, torch.arange(K, device=x.device)[None, :] < k[:, None])
    return dict(alpha=alpha, sg=sg, s=s, b=b, k=k, shared=shared, chosen=chosen, tau=tau)


def _expert_rows(case, r):
    """Each expert's tokens, their weights and which channels they run, in
    slices of at most 8,192 tokens."""
    M = case["H"] // case["B"]
    for e in range(case["K"] + 1):
        used = r["shared"].any(1) if e == 0 else r["chosen"][:, e - 1]
        for t in torch.split(used.nonzero().squeeze(1), 8192):
            if t.numel():
                w = r["alpha"][t] if e == 0 else r["s"][t, e - 1]
                blocks = r["shared"][t] if e == 0 else ~r["shared"][t]
                yield e, t, w[:, None], blocks.double().repeat_interleave(M, dim=1)


def exact(case, seed):
    device = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    v = _inputs(case, seed, device)
    T, d, H, K = case["T"], case["d"], case["H"], case["K"]
    valid = torch.ones(T, dtype=torch.bool, device=device) if v["mask"] is None else v["mask"] != 0
    x = v["x"].double()[valid]
    f = x
    if case["call"] == "sublayer":
        gamma, beta = v["gamma"].double(), v["beta"].double()
        if case["norm_first"]:  # LN(x) is kept in the layer dtype
            f = _layernorm(x, gamma, beta).to(v["x"].dtype).double()
    r = _route(case, v, f)
    y = torch.zeros_like(x)
    train = case["call"] == "train"
    if train:
        dy = v["dy"].double()[valid]
        dx, dwt = torch.zeros_like(x), torch.zeros(x.shape[0], K + 1, dtype=x.dtype, device=device)
        dw_up = torch.zeros(K + 1, H, d, dtype=x.dtype, device=device)
        dw_down = torch.zeros(K + 1, d, H, dtype=x.dtype, device=device)
    for e, t, w, keep in _expert_rows(case, r):
        wu, wd = v["w_up"][e].double(), v["w_down"][e].double()
        a = f[t] @ wu.T
        h = _gelu(a) * keep
        y.index_add_(0, t, w * (h @ wd.T))
        if train:
            g = (dy[t] @ wd) * keep
            dwt[t, e] += (h * g).sum(1)
            slope = 0.5 * (1 + torch.erf(a / math.sqrt(2.0))) \
                + a * torch.exp(-0.5 * a * a) / math.sqrt(2 * math.pi)
            da = w * g * slope
            dx.index_add_(0, t, da @ wu)
            dw_up[e] += da.T @ f[t]
            dw_down[e] += dy[t].T @ (w * h)
    if case["call"] == "sublayer":
        y = x + y
        if not case["norm_first"]:
            y = _layernorm(y, gamma, beta)

    def whole(u):
        out = torch.zeros(T, *u.shape[1:], dtype=u.dtype, device=device)
        out[valid] = u
        return out

    out = dict(y=whole(y), b=whole(r["b"].to(torch.int32)), k=whole(r["k"].to(torch.int32)))
    if train:
        dz = torch.zeros(x.shape[0], K + 1, dtype=x.dtype, device=device)
        if case["alpha_fixed"] < 0:
            dz[:, 0] = dwt[:, 0] * (1 - 2 * r["tau"]) * r["sg"] * (1 - r["sg"])
        dz[:, 1:] = r["s"] * (dwt[:, 1:] - (r["s"] * dwt[:, 1:]).sum(1, keepdim=True))
        wr = v["w_router"].double()
        gram = wr.T @ wr - torch.eye(K + 1, dtype=x.dtype, device=device)
        l_div = gram.norm()
        out.update(dx=whole(dx + dz @ wr.T), dw_up=dw_up, dw_down=dw_down,
                   dw_router=x.T @ dz + LAMBDA_DIV * 2 * wr @ gram / l_div, dbias=dz.sum(0),
                   l_div=l_div.reshape(1))
    return out
