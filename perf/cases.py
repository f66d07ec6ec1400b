"""Workloads by which the speed of the library is judged.

Each case is one pass through public entry points of
paper_2503_12450_gb300.lazymar, at the sizes of the repository's own
configurations (synth/inputs.py: MAR-B, MAR-L, MAR-H, high resolution and the
fp32 tiny model) or at ragged sizes of the same ranges:

  step      whole decoding steps: full, cached (both pathways), cached with the
            condition cache reused. The selected tokens of a cached step are
            fixed by priority classes, so that rounding cannot change them.
  linear    the four GEMMs of a block with their fused epilogues, over the rows
            of full layers, of recomputed tokens and of a few tokens
  e4m3      the 8-bit Q/K/V projection with its scatter into the token cache
  attention the subset and full-layer attention
  select    Eq. 8's token selection on two consecutive decoding steps
  layernorm the (optionally gathering) LayerNorm
  cfg       classifier-free guidance with the condition cache
  head      one call of the diffusion head: 100 denoising steps
"""
import math

import torch

from paper_2503_12450_gb300 import lazymar as lm

DEV = "cuda"
GAMMA = 3.0
EPS = 1e-6
KINDS = ("step", "linear", "e4m3", "attention", "select", "layernorm", "cfg", "head")

# transformer shapes: blocks, width, heads, buffer and image tokens, full blocks, dtype
MODELS = {
    "tiny": dict(depth=2, width=256, heads=4, n_buffer=16, n_img=64, sel_layers=1, dtype="fp32"),
    "mar_b": dict(depth=24, width=768, heads=12, n_buffer=64, n_img=256, sel_layers=3, dtype="bf16"),
    "mar_l": dict(depth=32, width=1024, heads=16, n_buffer=64, n_img=256, sel_layers=3, dtype="bf16"),
}
# denoiser shapes: width, residual blocks, width of z
HEADS = {
    "mar_b": dict(width=1024, depth=6, cond=768),
    "mar_l": dict(width=1280, depth=8, cond=1024),
    "mar_h": dict(width=1536, depth=12, cond=1280),
}
TOKEN_DIM, N_CLASSES, N_STEPS = 16, 1000, 100
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}
LM_DTYPES = {"fp32": lm.LAZYMAR_F32, "bf16": lm.LAZYMAR_BF16}
EPILOGUES = {"bias": lm.LAZYMAR_EPI_BIAS, "gelu": lm.LAZYMAR_EPI_GELU, "residual": lm.LAZYMAR_EPI_RESIDUAL,
             "qkv": lm.LAZYMAR_EPI_QKV}


def listed():
    return [
        # the smallest call a program makes: a cached step of the fp32 model, one pair
        dict(name="step-cached-tiny", kind="step", model="tiny", step="cached", batch=1, n=20, decoded=32),
        # the step most of a MAR-B decode consists of: 32 pairs, 50 of 320 tokens
        dict(name="step-cached-mar-b", kind="step", model="mar_b", step="cached", batch=32, n=50, decoded=60),
        # a refresh step of a MAR-L decode
        dict(name="step-full-mar-l", kind="step", model="mar_l", step="full", batch=32, n=0, decoded=120),
        # Q/K/V projection of the recomputed tokens, scattered into the token cache
        dict(name="qkv-recomputed", kind="linear", role="qkv", dtype="bf16", rows=64, n=50, T=320, D=768),
        # MLP up-projection with GELU over a full layer
        dict(name="fc1-full", kind="linear", role="fc1", dtype="bf16", rows=64, n=320, T=320, D=768),
        # MLP down-projection into the residual stream on a condition-reuse step
        dict(name="fc2-reuse", kind="linear", role="fc2", dtype="bf16", rows=32, n=50, T=320, D=768),
        # attention output projection at the widest model, a ragged number of rows
        dict(name="out-ragged", kind="linear", role="out", dtype="bf16", rows=7, n=143, T=320, D=1280),
        # recomputed tokens attending over all tokens
        dict(name="attention-subset", kind="attention", rows=64, n=50, T=320, heads=12, dh=64),
        # full-layer attention with heads of 80
        dict(name="attention-full-80", kind="attention", rows=64, n=320, T=320, heads=16, dh=80),
        # token selection of a cached step, on two consecutive steps
        dict(name="select", kind="select", dtype="bf16", rows=64, T=320, D=768, n=50),
        # LayerNorm of the recomputed tokens
        dict(name="layernorm", kind="layernorm", dtype="bf16", M=3200, D=768, gather=False),
        # the latents of 4 new tokens of each of 32 pairs
        dict(name="head-sample", kind="head", model="mar_b", pairs=32, new=4, n_img=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "linear", "linear", "linear", "linear", "e4m3", "attention", "attention",
                       "attention", "select", "select", "layernorm", "cfg", "head", "head"])
    if kind == "step":
        model = rng.choice(["tiny", "mar_b", "mar_b", "mar_l"])
        batch = {"tiny": _log(rng, 1, 8), "mar_b": _log(rng, 1, 32), "mar_l": _log(rng, 1, 16)}[model]
        m = MODELS[model]
        T = m["n_buffer"] + m["n_img"]
        return dict(kind=kind, model=model, step=rng.choice(["full", "cached", "cached", "reuse"]), batch=batch,
                    n=rng.randint(T // 8, T // 3), decoded=rng.randint(m["n_img"] // 8, m["n_img"] - 8))
    if kind == "linear":
        role = rng.choice(["qkv", "out", "fc1", "fc2"])
        if rng.random() < 0.15:  # the fp32 model
            return dict(kind=kind, role=role, dtype="fp32", rows=rng.randint(1, 8), n=rng.randint(8, 80), T=80, D=256)
        T = rng.choice([320, 1088])
        n = T if rng.random() < 0.4 else rng.randint(1, T // 2)
        return dict(kind=kind, role=role, dtype="bf16", rows=_log(rng, 1, 64 if T == 320 else 16), n=n, T=T,
                    D=rng.choice([768, 1024, 1280]))
    if kind == "e4m3":
        return dict(kind=kind, rows=_log(rng, 1, 64), n=rng.randint(16, 160), T=320, D=rng.choice([768, 1024, 1280]))
    if kind == "attention":
        T = rng.choice([320, 320, 1088, rng.randint(65, 700)])
        heads, dh = rng.choice([(12, 64), (16, 64), (16, 80)])
        n = T if rng.random() < 0.4 else rng.randint(1, T // 2)
        return dict(kind=kind, rows=_log(rng, 1, 64 if T <= 320 else 16), n=n, T=T, heads=heads, dh=dh)
    if kind == "select":
        T = rng.choice([320, 1088, rng.randint(65, 1088)])
        return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "fp32"]), rows=_log(rng, 1, 64 if T <= 320 else 24),
                    T=T, D=rng.choice([768, 1024, 1280]), n=rng.randint(1, T // 2))
    if kind == "layernorm":
        return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "fp32"]), M=_log(rng, 16, 40960),
                    D=rng.choice([256, 768, 1024, 1280]), gather=rng.random() < 0.3)
    if kind == "cfg":
        return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "fp32"]), mode=rng.choice(["refresh", "reuse"]),
                    pairs=_log(rng, 1, 64), n_img=256, D=rng.choice([768, 1024, 1280]))
    model = rng.choice(["mar_b", "mar_b", "mar_l", "mar_h"])
    return dict(kind="head", model=model, pairs=_log(rng, 1, 32), new=rng.randint(1, 7), n_img=256)


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, std=1.0, mean=0.0):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32) * std + mean


def _perm(g, rows, T, n):
    """n distinct tokens of each of `rows` rows, ascending."""
    return torch.rand((rows, T), generator=g, device=DEV).argsort(dim=1)[:, :n].sort(dim=1).values


def _model_weights(m, g):
    """Random weights ([out, in] layout), representable in the model's dtype."""
    D, T = m["width"], m["n_buffer"] + m["n_img"]

    def w(*shape, std=0.02, mean=0.0):
        x = _normal(g, shape, std, mean)
        return x.bfloat16().float() if m["dtype"] == "bf16" else x

    W = dict(pos_emb=w(T, D), class_emb=w(N_CLASSES, D), mask_emb=w(D), embed_w=w(D, TOKEN_DIM), embed_b=w(D),
             lnf_g=w(D, std=0.1, mean=1.0), lnf_b=w(D), blocks=[])
    for _ in range(m["depth"]):
        W["blocks"].append(dict(
            ln1_g=w(D, std=0.1, mean=1.0), ln1_b=w(D), w_qkv=w(3 * D, D), b_qkv=w(3 * D), w_o=w(D, D), b_o=w(D),
            ln2_g=w(D, std=0.1, mean=1.0), ln2_b=w(D), w1=w(4 * D, D), b1=w(4 * D), w2=w(D, 4 * D), b2=w(D)))
    return W


def _head_weights(hc, g):
    w, c = hc["width"], hc["cond"]

    def r(*shape):
        return _normal(g, shape, 0.02).bfloat16().float()

    W = dict(t_w1=r(w, 256), t_b1=r(w), t_w2=r(w, w), t_b2=r(w), c_w=r(w, c), c_b=r(w), in_w=r(w, TOKEN_DIM), in_b=r(w),
             blocks=[dict(ada_w=r(3 * w, w), ada_b=r(3 * w), w1=r(w, w), b1=r(w), w2=r(w, w), b2=r(w))
                     for _ in range(hc["depth"])])
    W.update(f_ada_w=r(2 * w, w), f_ada_b=r(2 * w), out_w=r(2 * TOKEN_DIM, w), out_b=r(2 * TOKEN_DIM))
    return W


def _step_rows(c):
    return c["batch"] if c["step"] == "reuse" else 2 * c["batch"]


def _step_inputs(c, seed):
    """Weights and the inputs of two consecutive decoding steps: the step that
    fills the caches, then the step of the case with 8 more decoded tokens."""
    m = MODELS[c["model"]]
    g = _gen(seed)
    B, n_img, T = c["batch"], m["n_img"], m["n_buffer"] + m["n_img"]
    W = _model_weights(m, g)
    labels = torch.randint(0, N_CLASSES, (B,), generator=g, device=DEV, dtype=torch.int32)
    table = _normal(g, (B, n_img, TOKEN_DIM))
    rank = torch.rand((B, n_img), generator=g, device=DEV).argsort(dim=1).argsort(dim=1)
    ins = []
    for decoded in (c["decoded"] - 8, c["decoded"]):
        mask = (rank >= decoded)
        ins.append((torch.where(mask[..., None], torch.zeros_like(table), table).contiguous(),
                    mask.to(torch.uint8).contiguous()))
    idx = None
    if c["step"] != "full":
        idx = _perm(g, _step_rows(c), T, c["n"])
    return m, W, labels, ins, idx


def _linear_dims(c):
    D = c["D"]
    return {"qkv": (3 * D, D, "qkv"), "out": (D, D, "residual"), "fc1": (4 * D, D, "gelu"),
            "fc2": (D, 4 * D, "residual")}[c["role"]]


def _linear_inputs(c, seed):
    N, K, epi = _linear_dims(c)
    g = _gen(seed)
    M, D = c["rows"] * c["n"], c["D"]
    dt = DTYPES[c["dtype"]]
    x = dict(a=_normal(g, (M, K), 1.0 if c["role"] != "fc2" else 0.3).to(dt), w=_normal(g, (N, K), 0.02).to(dt),
             b=_normal(g, (N,), 0.02).to(dt))
    if epi == "residual":
        x["out"] = _normal(g, (M, N))
    elif epi == "gelu":
        x["out"] = torch.empty((M, N), device=DEV, dtype=dt)
    else:
        x["out"] = torch.empty((M, D), device=DEV, dtype=dt)
        # the token cache: fresh keys and values go to the rows of their tokens
        x["k"] = _normal(g, (c["rows"] * c["T"], D)).to(dt)
        x["v"] = _normal(g, (c["rows"] * c["T"], D)).to(dt)
        x["map"] = None
        if c["n"] < c["T"]:
            sel = _perm(g, c["rows"], c["T"], c["n"])
            x["map"] = (sel + torch.arange(c["rows"], device=DEV)[:, None] * c["T"]).reshape(-1).int().contiguous()
    return x


def _e4m3_inputs(c, seed):
    g = _gen(seed)
    M, D = c["rows"] * c["n"], c["D"]
    sel = _perm(g, c["rows"], c["T"], c["n"])
    return dict(a=_normal(g, (M, D)).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8),
                w=_normal(g, (3 * D, D), 0.02).bfloat16(), b=_normal(g, (3 * D,), 0.02).bfloat16(),
                out=torch.empty((M, D), device=DEV, dtype=torch.bfloat16),
                k=_normal(g, (c["rows"] * c["T"], D)).bfloat16(), v=_normal(g, (c["rows"] * c["T"], D)).bfloat16(),
                map=(sel + torch.arange(c["rows"], device=DEV)[:, None] * c["T"]).reshape(-1).int().contiguous())


def _attention_inputs(c, seed):
    g = _gen(seed)
    D = c["heads"] * c["dh"]
    return dict(q=_normal(g, (c["rows"], c["n"], D)).bfloat16(), k=_normal(g, (c["rows"], c["T"], D)).bfloat16(),
                v=_normal(g, (c["rows"], c["T"], D)).bfloat16(),
                o=torch.empty((c["rows"], c["n"], D), device=DEV, dtype=torch.bfloat16))


def _select_inputs(c, seed):
    """Values of two consecutive steps: most tokens move a little between them,
    one in ten (those just decoded) a lot."""
    g = _gen(seed)
    shape = (c["rows"], c["T"], c["D"])
    a = _normal(g, shape, 0.5)
    moved = torch.rand(shape[:2], generator=g, device=DEV) < 0.1
    small = 0.005 + 0.05 * torch.rand(shape[:2], generator=g, device=DEV)
    b = torch.where(moved[..., None], _normal(g, shape, 0.5), a + small[..., None] * _normal(g, shape, 0.5))
    dt = DTYPES[c["dtype"]]
    return a.to(dt), b.to(dt)


def _layernorm_inputs(c, seed):
    g = _gen(seed)
    dt = DTYPES[c["dtype"]]
    src = 4 * c["M"] if c["gather"] else c["M"]
    return dict(x=_normal(g, (src, c["D"]), 2.0, 0.3), g=_normal(g, (c["D"],), 0.1, 1.0).to(dt),
                b=_normal(g, (c["D"],), 0.02).to(dt),
                map=torch.randperm(src, generator=g, device=DEV)[:c["M"]].int().contiguous() if c["gather"] else None,
                y=torch.empty((c["M"], c["D"]), device=DEV, dtype=dt))


def _cfg_inputs(c, seed):
    g = _gen(seed)
    n, dt = c["pairs"] * c["n_img"] * c["D"], DTYPES[c["dtype"]]
    z = _normal(g, (n,))
    return dict(zc=z.to(dt), zu=(z + 0.3 * _normal(g, (n,))).to(dt), d=(0.3 * _normal(g, (n,))).to(dt),
                uo=torch.empty((n,), device=DEV, dtype=dt), g=torch.empty((n,), device=DEV, dtype=dt), n=n)


def _head_inputs(c, seed):
    hc = HEADS[c["model"]]
    g = _gen(seed)
    M = c["pairs"] * c["new"]
    W = _head_weights(hc, g)
    z = _normal(g, (2 * c["pairs"], c["n_img"], hc["cond"])).bfloat16()
    pos = _perm(g, c["pairs"], c["n_img"], c["new"]).int().contiguous()
    noise = _normal(g, (N_STEPS, M, TOKEN_DIM))
    return hc, W, z, pos, noise, M


def prepare(case, seed):
    c = case
    if c["kind"] == "step":
        m, W, labels, ins, idx = _step_inputs(c, seed)
        B, T = c["batch"], m["n_buffer"] + m["n_img"]
        h = lm.lazymar_create(dict(m, mlp_ratio=4, token_dim=TOKEN_DIM, n_classes=N_CLASSES, max_batch=B, ln_eps=EPS),
                              W)
        dt = DTYPES[m["dtype"]]
        s = dict(c=c, h=h, labels=labels, lat=ins[1][0], mask=ins[1][1],
                 z=torch.empty((2 * B, m["n_img"], m["width"]), device=DEV, dtype=dt),
                 g=torch.empty((B, m["n_img"], m["width"]), device=DEV, dtype=dt))
        if c["step"] != "full":
            s["prio"] = torch.zeros((_step_rows(c), T), device=DEV, dtype=torch.uint8).scatter_(1, idx, 1)
            s["idx"] = torch.empty((_step_rows(c), c["n"]), device=DEV, dtype=torch.int32)
            lm.lazymar_full_step(h, ins[0][0], ins[0][1], labels, B, GAMMA)
            torch.cuda.synchronize()
        return s
    if c["kind"] == "linear":
        return dict(c=c, **_linear_inputs(c, seed))
    if c["kind"] == "e4m3":
        s = dict(c=c, **_e4m3_inputs(c, seed))
        s["q8"] = torch.empty(s["w"].shape, device=DEV, dtype=torch.uint8)
        s["sc"] = torch.empty((3 * c["D"],), device=DEV, dtype=torch.float32)
        lm.lazymar_quantize_e4m3(s["w"], 3 * c["D"], c["D"], s["q8"], s["sc"])
        return s
    if c["kind"] == "attention":
        return dict(c=c, **_attention_inputs(c, seed))
    if c["kind"] == "select":
        a, b = _select_inputs(c, seed)
        return dict(c=c, a=a, b=b, cache=b.clone(),
                    i1=torch.empty((c["rows"], c["n"]), device=DEV, dtype=torch.int32),
                    i2=torch.empty((c["rows"], c["n"]), device=DEV, dtype=torch.int32))
    if c["kind"] == "layernorm":
        return dict(c=c, **_layernorm_inputs(c, seed))
    if c["kind"] == "cfg":
        return dict(c=c, **_cfg_inputs(c, seed))
    hc, W, z, pos, noise, M = _head_inputs(c, seed)
    hd = lm.lazymar_head_create(dict(width=hc["width"], depth=hc["depth"], freq_dim=256, n_train=1000,
                                     n_steps=N_STEPS), hc["cond"], TOKEN_DIM, W, max_tokens=M)
    return dict(c=c, hd=hd, z=z, pos=pos, noise=noise, x=torch.empty((M, TOKEN_DIM), device=DEV))


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "step":
        if c["step"] == "full":
            lm.lazymar_full_step(s["h"], s["lat"], s["mask"], s["labels"], c["batch"], GAMMA, s["z"], s["g"])
            return dict(z=s["z"], guided=s["g"])
        lm.lazymar_cached_step(s["h"], s["lat"], s["mask"], s["labels"], c["batch"], c["n"], c["step"] == "reuse",
                               GAMMA, idx_out=s["idx"], z_out=s["z"], guided_out=s["g"], select_priority=s["prio"])
        return dict(z=s["z"], guided=s["g"], idx=s["idx"])
    if kind == "linear":
        N, K, epi = _linear_dims(c)
        M = c["rows"] * c["n"]
        if epi == "qkv":
            lm.lazymar_linear(LM_DTYPES[c["dtype"]], EPILOGUES[epi], s["a"], s["w"], s["b"], M, N, K, s["out"], c["D"],
                              s["k"], s["v"], s["map"])
            return dict(q=s["out"], k=s["k"], v=s["v"])
        lm.lazymar_linear(LM_DTYPES[c["dtype"]], EPILOGUES[epi], s["a"], s["w"], s["b"], M, N, K, s["out"], N)
        return s["out"]
    if kind == "e4m3":
        lm.lazymar_linear_e4m3(lm.LAZYMAR_EPI_QKV, s["a"], s["q8"], s["sc"], s["b"], c["rows"] * c["n"], 3 * c["D"],
                               c["D"], s["out"], c["D"], s["k"], s["v"], s["map"])
        return dict(q=s["out"], k=s["k"], v=s["v"])
    if kind == "attention":
        lm.lazymar_attention(lm.LAZYMAR_BF16, s["q"], s["k"], s["v"], s["o"], c["rows"], c["n"], c["T"], c["heads"],
                             c["dh"])
        return s["o"]
    if kind == "select":
        dt = LM_DTYPES[c["dtype"]]
        lm.lazymar_select_tokens(dt, s["a"], s["cache"], c["rows"], c["T"], c["D"], c["n"], s["i1"])
        lm.lazymar_select_tokens(dt, s["b"], s["cache"], c["rows"], c["T"], c["D"], c["n"], s["i2"])
        return dict(first=s["i1"], second=s["i2"], cache=s["cache"])
    if kind == "layernorm":
        lm.lazymar_layernorm(LM_DTYPES[c["dtype"]], s["x"], s["map"], s["g"], s["b"], s["y"], c["M"], c["D"], EPS)
        return s["y"]
    if kind == "cfg":
        dt = LM_DTYPES[c["dtype"]]
        if c["mode"] == "refresh":
            lm.lazymar_cfg_combine(dt, lm.LAZYMAR_CFG_REFRESH, s["zc"], s["zu"], s["d"], GAMMA, s["n"], None, s["g"])
            return dict(delta=s["d"], guided=s["g"])
        lm.lazymar_cfg_combine(dt, lm.LAZYMAR_CFG_REUSE, s["zc"], None, s["d"], GAMMA, s["n"], s["uo"], s["g"])
        return dict(uncond=s["uo"], guided=s["g"])
    lm.lazymar_head_sample(s["hd"], s["z"], c["pairs"], c["n_img"], s["pos"], c["new"], s["noise"], GAMMA, 1.0, s["x"])
    return s["x"]


# ----------------------------------------------------------------------------
# Work
# ----------------------------------------------------------------------------
def work(case):
    c = case
    kind = c["kind"]
    if kind == "step":
        m = MODELS[c["model"]]
        D, L, sl, T = m["width"], m["depth"], m["sel_layers"], m["n_buffer"] + m["n_img"]
        es = 2 if m["dtype"] == "bf16" else 4
        B, rows = c["batch"], _step_rows(c)
        io = B * m["n_img"] * (TOKEN_DIM * 4 + 1) + 3 * B * m["n_img"] * D * es
        weights = L * 12 * D * D * es
        if c["step"] == "full":
            M = rows * T
            return dict(flops=L * (24.0 * M * D * D + 4.0 * M * T * D),
                        bytes=weights + io + 2.0 * (L - sl) * M * D * es + M * D * es)
        M, Mc = rows * T, rows * c["n"]
        flops = (sl - 1) * (24.0 * M * D * D + 4.0 * M * T * D) + 6.0 * M * D * D + 18.0 * Mc * D * D
        flops += (L - sl) * 24.0 * Mc * D * D + (L - sl + 1) * 4.0 * Mc * T * D
        return dict(flops=flops, bytes=weights + io + 2.0 * (L - sl) * M * D * es + 2.0 * M * D * es)
    if kind == "linear":
        N, K, epi = _linear_dims(c)
        M, es = c["rows"] * c["n"], 2 if c["dtype"] == "bf16" else 4
        return dict(flops=2.0 * M * N * K, bytes=es * (M * K + N * K + N) + (8.0 if epi == "residual" else es) * M * N)
    if kind == "e4m3":
        M, D = c["rows"] * c["n"], c["D"]
        return dict(flops=6.0 * M * D * D, bytes=M * D + 3.0 * D * D + 6.0 * M * D)
    if kind == "attention":
        D = c["heads"] * c["dh"]
        return dict(flops=4.0 * c["rows"] * c["n"] * c["T"] * D, bytes=4.0 * c["rows"] * D * (c["T"] + c["n"]))
    if kind == "select":
        es = 2 if c["dtype"] == "bf16" else 4
        return dict(flops=2 * 6.0 * c["rows"] * c["T"] * c["D"], bytes=2 * 3.0 * es * c["rows"] * c["T"] * c["D"])
    if kind == "layernorm":
        return dict(flops=0.0, bytes=c["M"] * c["D"] * (4.0 + (2 if c["dtype"] == "bf16" else 4)))
    if kind == "cfg":
        return dict(flops=0.0, bytes=4.0 * (2 if c["dtype"] == "bf16" else 4) * c["pairs"] * c["n_img"] * c["D"])
    hc = HEADS[c["model"]]
    w, R = hc["width"], 2 * c["pairs"] * c["new"]
    mod = 3 * w * hc["depth"] + 2 * w
    per = 2.0 * R * w * (mod + 2 * hc["depth"] * w + 3 * TOKEN_DIM)
    return dict(flops=N_STEPS * per + 2.0 * R * w * hc["cond"],
                bytes=2.0 * w * (mod + 2 * hc["depth"] * w + hc["cond"]) + R * hc["cond"] * 2.0 +
                N_STEPS * R / 2 * TOKEN_DIM * 4.0)


# ----------------------------------------------------------------------------
# Tolerances and the same in 64 bits
# ----------------------------------------------------------------------------
def tolerance(case):
    """About four times the largest error against `exact` that was seen over the listed and drawn cases: "rel" of the
    2-norm, "max" of one value."""
    c = case
    kind = c["kind"]
    if kind == "select":  # token indices and copied values
        return "exact"
    if kind == "step":
        # bf16: guided = u + 3 (c - u) triples the features' error (4e-3 of z, 1.1e-2 of guided)
        return dict(rel=1e-5, max=1e-4) if c["model"] == "tiny" else dict(rel=3e-2, max=0.25)
    if kind == "head":  # 100 bf16 network evaluations in a chain
        return dict(rel=2.5e-2, max=0.1)
    if c.get("dtype") == "fp32" or (kind == "linear" and _linear_dims(c)[2] == "residual"):  # fp32 results
        return dict(rel=6e-6, max=1e-4)
    if kind == "attention":  # bf16 probabilities and results
        return dict(rel=1e-2, max=6e-2)
    if kind == "e4m3":
        return dict(rel=1e-2, max=0.25)
    return dict(rel=7e-3, max=1.6e-2)  # one rounding to bf16


def _ln(x, g=None, b=None):
    mu = x.mean(-1, keepdim=True)
    v = ((x - mu) ** 2).mean(-1, keepdim=True)
    y = (x - mu) / torch.sqrt(v + EPS)
    return y if g is None else y * g.double() + b.double()


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _silu(x):
    return x / (1.0 + torch.exp(-x))


def _lin(x, w, b):
    return x @ w.double().T + b.double()


def _attend(q, k, v, heads):
    R, n, D = q.shape
    T, dh = k.shape[1], D // heads
    out = torch.empty_like(q)
    step = max(1, int(3e8 // (heads * n * T)))
    for r in range(0, R, step):
        qq, kk, vv = (x[r:r + step].reshape(-1, x.shape[1], heads, dh).transpose(1, 2) for x in (q, k, v))
        p = torch.softmax(qq @ kk.transpose(2, 3) / math.sqrt(dh), dim=-1)
        out[r:r + step] = (p @ vv).transpose(1, 2).reshape(-1, n, D)
    return out


def _exact_step(c, seed):
    m, W, labels, ins, idx = _step_inputs(c, seed)
    D, L, sl, nb = m["width"], m["depth"], m["sel_layers"], m["n_buffer"]
    H, B = m["heads"], c["batch"]

    def embed(lat, mask, both):
        img = _lin(lat.double(), W["embed_w"], W["embed_b"])
        img = torch.where(mask[..., None] != 0, W["mask_emb"].double(), img)
        buf = W["class_emb"].double()[labels.long()][:, None, :].expand(-1, nb, -1)
        rows = [torch.cat([buf, img], 1)]
        if both:
            rows.append(torch.cat([torch.zeros_like(buf), img], 1))
        return torch.cat(rows, 0) + W["pos_emb"].double()

    def qkv(w, x):
        y = _lin(_ln(x, w["ln1_g"], w["ln1_b"]), w["w_qkv"], w["b_qkv"])
        return y[..., :D], y[..., D:2 * D], y[..., 2 * D:]

    def rest(w, x, o):
        y = x + _lin(o, w["w_o"], w["b_o"])
        return y + _lin(_gelu(_lin(_ln(y, w["ln2_g"], w["ln2_b"]), w["w1"], w["b1"])), w["w2"], w["b2"])

    def full(lat, mask):
        x = embed(lat, mask, True)
        kv = []
        for w in W["blocks"]:
            q, k, v = qkv(w, x)
            kv.append((k, v))
            x = rest(w, x, _attend(q, k, v, H))
        return x, kv

    def final(x):
        return _ln(x[:, nb:], W["lnf_g"], W["lnf_b"])

    if c["step"] == "full":
        z = final(full(*ins[1])[0])
        return dict(z=z, guided=z[B:] + GAMMA * (z[:B] - z[B:]))
    last, kv = full(*ins[0])
    z0 = final(last)
    delta = z0[:B] - z0[B:]
    R = _step_rows(c)
    x = embed(*ins[1], R == 2 * B)
    for w in W["blocks"][:sl]:
        q, k, v = qkv(w, x)
        x = rest(w, x, _attend(q, k, v, H))
    sel = idx[..., None].expand(-1, -1, D)
    xs = torch.gather(x, 1, sel)
    for l in range(sl, L):
        w = W["blocks"][l]
        q, k, v = qkv(w, xs)
        K, V = kv[l][0][:R].scatter(1, sel, k), kv[l][1][:R].scatter(1, sel, v)
        xs = rest(w, xs, _attend(q, K, V, H))
    z = final(last[:R].scatter(1, sel, xs))
    if R == B:
        z = torch.cat([z, z - delta], 0)
    return dict(z=z, guided=z[B:] + GAMMA * (z[:B] - z[B:]), idx=None)


def _alpha_bars(n_train):
    f = [math.cos((t / n_train + 0.008) / 1.008 * math.pi / 2) ** 2 for t in range(n_train + 1)]
    ab, p = [], 1.0
    for t in range(n_train):
        p *= 1.0 - min(1.0 - f[t + 1] / f[t], 0.999)
        ab.append(p)
    return ab


def _exact_head(c, seed):
    hc, W, z, pos, noise, M = _head_inputs(c, seed)
    w, depth = hc["width"], hc["depth"]
    W = {k: ([{n: x.double() for n, x in b.items()} for b in v] if k == "blocks" else v.double()) for k, v in W.items()}
    B = c["pairs"]
    at = pos.long()[..., None].expand(-1, -1, hc["cond"])
    zz = torch.cat([torch.gather(z[:B].double(), 1, at).reshape(M, -1),
                    torch.gather(z[B:].double(), 1, at).reshape(M, -1)], 0)
    cemb = _lin(zz, W["c_w"], W["c_b"])
    ab = _alpha_bars(1000)
    kept = [int(round(i * 999 / (N_STEPS - 1))) for i in range(N_STEPS)]
    abk = [ab[t] for t in kept]
    x = noise[0].double()
    for i in range(N_STEPS):
        j = N_STEPS - 1 - i
        fr = torch.exp(-math.log(10000.0) * torch.arange(128, device=DEV, dtype=torch.float64) / 128) * kept[j]
        t = _lin(_silu(_lin(torch.cat([torch.cos(fr), torch.sin(fr)])[None], W["t_w1"], W["t_b1"])), W["t_w2"], W["t_b2"])
        sy = _silu(t + cemb)
        h = _lin(torch.cat([x, x], 0), W["in_w"], W["in_b"])
        for b in W["blocks"]:
            sh, sc, ga = _lin(sy, b["ada_w"], b["ada_b"]).split(w, 1)
            h = h + ga * _lin(_silu(_lin(_ln(h) * (1 + sc) + sh, b["w1"], b["b1"])), b["w2"], b["b2"])
        sh, sc = _lin(sy, W["f_ada_w"], W["f_ada_b"]).split(w, 1)
        o = _lin(_ln(h) * (1 + sc) + sh, W["out_w"], W["out_b"])
        e = o[M:, :TOKEN_DIM] + GAMMA * (o[:M, :TOKEN_DIM] - o[M:, :TOKEN_DIM])
        a, pa = abk[j], abk[j - 1] if j else 1.0
        beta = 1.0 - a / pa
        x0 = x / math.sqrt(a) - math.sqrt(1.0 / a - 1.0) * e
        x = beta * math.sqrt(pa) / (1 - a) * x0 + (1 - pa) * math.sqrt(1 - beta) / (1 - a) * x
        if j:
            post = beta * (1 - pa) / (1 - a)
            frac = (o[:M, TOKEN_DIM:] + 1) / 2
            x = x + torch.exp(0.5 * (frac * math.log(beta) + (1 - frac) * math.log(post))) * noise[i + 1].double()
    return x


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "step":
        return _exact_step(c, seed) if work(c)["flops"] < 2.5e13 else None
    if kind == "head":
        return _exact_head(c, seed) if work(c)["flops"] < 2.5e13 else None
    if kind == "linear":
        x = _linear_inputs(c, seed)
        y = _lin(x["a"].double(), x["w"], x["b"])
        epi = _linear_dims(c)[2]
        if epi == "qkv":
            return _scattered(c, x, y)
        return _gelu(y) if epi == "gelu" else x["out"].double() + y
    if kind == "e4m3":
        x = _e4m3_inputs(c, seed)
        w = x["w"].float()
        s = w.abs().amax(1, keepdim=True) / 448.0
        q = (w / s).to(torch.float8_e4m3fn).double() * s.double()
        return _scattered(c, x, _lin(x["a"].view(torch.float8_e4m3fn).double(), q, x["b"]))
    if kind == "attention":
        x = _attention_inputs(c, seed)
        return _attend(x["q"].double(), x["k"].double(), x["v"].double(), c["heads"])
    if kind == "select":
        b = _select_inputs(c, seed)[1]
        return dict(first=None, second=None, cache=b.double())
    if kind == "layernorm":
        x = _layernorm_inputs(c, seed)
        src = x["x"].double()
        return _ln(src if x["map"] is None else src[x["map"].long()], x["g"], x["b"])
    x = _cfg_inputs(c, seed)
    z, u, d = x["zc"].double(), x["zu"].double(), x["d"].double()
    if c["mode"] == "refresh":
        return dict(delta=z - u, guided=u + GAMMA * (z - u))
    return dict(uncond=z - d, guided=(z - d) + GAMMA * d)


def _scattered(c, x, y):
    D = c["D"]
    k, v = x["k"].double(), x["v"].double()
    at = torch.arange(y.shape[0], device=DEV) if x["map"] is None else x["map"].long()
    k[at], v[at] = y[:, D:2 * D], y[:, 2 * D:]
    return dict(q=y[:, :D].contiguous(), k=k, v=v)
