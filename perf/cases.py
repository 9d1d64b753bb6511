"""The work that is timed when this library's speed is looked at: what a user has it do, through its public
entry points, from a single small layer to whole networks at full batch.

Kinds of case
  layer     one masked convolution (bf16, or quantised to e4m3 first; plain, with a skip connection, grouped)
  resnet    forward pass of the ResNet-50-shaped stack (stack.ConvStack) on raw RGB images, skip connections fused
  convnext  forward pass of the ConvNeXt-T-shaped network (convnext.ConvNeXtStack) on raw RGB images
  train     one mask-learning step of one layer: soft mask, dense forward with the effective weights, weight and
            input gradient, gradient of the choice weights, AdamW
  masks     what loading a network costs: choose and pack the masks of all 52 masked layers of the ResNet-50 stack
"""
import dataclasses
import math

import torch

from paper_2411_00288_b200 import api, convnext, stack, synth

DEV = "cuda:0"
TAU = 0.5                        # temperature of the relaxed choice, as in the benchmark's mask-learning step
W_SCALE = 16.0                   # scale of e4m3 weights, as in the benchmark's 8-bit leg


def _layer(name, n, h, w, cin, cout, k, stride, pad, act="relu", res=False, dtype="bf16", groups=1):
    return dict(name=name, kind="layer", n=n, h=h, w=w, cin=cin, cout=cout, k=k, stride=stride, pad=pad, act=act, res=res,
                dtype=dtype, groups=groups)


def _train(name, n, h, w, cin, cout, k, stride, pad):
    return dict(name=name, kind="train", n=n, h=h, w=w, cin=cin, cout=cout, k=k, stride=stride, pad=pad)


def listed():
    return [
        # one layer on one image (the first workload configuration): a call's latency
        _layer("layer_3x3_c64_b1", 1, 14, 14, 64, 64, 3, 1, 1),
        # a layer of the stack on 8-bit operands, activations quantised on the way in
        _layer("layer_e4m3_3x3_c256_b256", 256, 14, 14, 256, 256, 3, 1, 1, dtype="e4m3"),
        # a grouped convolution (few wide groups), ragged output channels
        _layer("layer_grouped_3x3_b64", 64, 14, 14, 256, 288, 3, 1, 1, groups=4),
        # online inference: one image through the network
        dict(name="resnet50_b1", kind="resnet", batch=1),
        # a serving batch that fills no tile exactly
        dict(name="resnet50_b27", kind="resnet", batch=27),
        # the benchmark's batch: offline inference
        dict(name="resnet50_b256", kind="resnet", batch=256),
        # the other network family, a few images and the benchmark's batch
        dict(name="convnext_t_b3", kind="convnext", batch=3, image=224),
        dict(name="convnext_t_b128", kind="convnext", batch=128, image=224),
        # learning the masks: a 3x3 layer, a strided one, a wide pointwise one
        _train("train_3x3_c256_b64", 64, 14, 14, 256, 256, 3, 1, 1),
        _train("train_3x3s2_c128_b32", 32, 28, 28, 128, 256, 3, 2, 1),
        _train("train_1x1_c96_b128", 128, 56, 56, 96, 384, 1, 1, 0),
        # choosing and packing a whole network's masks from learned choice weights
        dict(name="masks_resnet50", kind="masks", width=64),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _channels(rng, lo, hi, step=8):
    return max(lo, _log_int(rng, lo, hi) // step * step)


def draw(rng):
    have = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        c = _draw(rng)
        if c not in have:
            return c


def _draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "resnet", "convnext", "train", "train", "masks"])
    if kind == "resnet":
        return dict(kind=kind, batch=_log_int(rng, 1, 250))
    if kind == "convnext":
        image = 32 * rng.randint(3, 8)
        most = min(256, int(128 * 224 * 224 / image ** 2))
        return dict(kind=kind, batch=_log_int(rng, 1, most), image=image)
    if kind == "masks":
        return dict(kind=kind, width=8 * rng.randint(2, 12))
    while True:
        k = rng.choice([1, 1, 3, 3, 3, 5])
        stride = rng.choice([1, 1, 1, 2])
        pad = rng.randint(0, k // 2)
        h = _log_int(rng, 7, 64)
        w = h if rng.random() < 0.7 else _log_int(rng, 7, 64)
        n = _log_int(rng, 1, 256)
        dtype = "e4m3" if kind == "layer" and rng.random() < 0.25 else "bf16"
        step = 16 if dtype == "e4m3" else 8
        cin, cout = _channels(rng, 16, 2048, step), _channels(rng, 16, 2048)
        groups = 1
        if kind == "layer" and dtype == "bf16" and rng.random() < 0.2:
            groups = rng.choice([2, 3, 4])
            cin, cout = groups * _channels(rng, 16, 256), groups * _channels(rng, 16, 256)
        c = _layer("", n, h, w, cin, cout, k, stride, pad, dtype=dtype, groups=groups) if kind == "layer" else _train(
            "", n, h, w, cin, cout, k, stride, pad)
        del c["name"]
        if kind == "layer":
            c["act"] = rng.choice(["relu", "relu", "gelu", "none"])
            c["res"] = groups == 1 and dtype == "bf16" and rng.random() < 0.3
        if work(c)["flops"] <= 1.0e12 and work(c)["bytes"] <= 3.0e9:   # below the largest listed case
            return c


# ----------------------------------------------------------------------------- what a user has in hand
def _desc(c):
    act = c.get("act", "none")
    return api.make_desc(c["n"], c["h"], c["w"], c["cin"], c["cout"], c["k"], c["k"], stride=c["stride"], pad=c["pad"],
                         bias=True, relu=act == "relu", gelu=act == "gelu")


def _extent(c):
    return ((c["h"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1, (c["w"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1)


def _randn(g, *shape, std=1.0, dtype=torch.bfloat16):
    return (torch.randn(shape, generator=g, device=DEV, dtype=torch.float32) * std).to(dtype)


def _gumbel(g, *shape):
    u = torch.rand(shape, generator=g, device=DEV, dtype=torch.float32).clamp_(1e-6, 1.0 - 1e-6)
    return -torch.log(-torch.log(u))


def _resnet_steps(batch, seed):
    # the stack's own layer list, its seeded weights moved to other draws for other seeds
    return [st if st.spec is None else dataclasses.replace(st, spec=dataclasses.replace(st.spec, index=st.spec.index + 1000 * (seed % 997)))
            for st in synth.resnet50_stack(batch, residual=True)]


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "resnet":
        s["x"] = _randn(g, case["batch"], 224, 224, 3)
        s["net"] = stack.ConvStack(_resnet_steps(case["batch"], seed), DEV)
        # the last block of each stage: the feature maps a user of a backbone reads
        s["taps"] = [i for i, st in enumerate(s["net"].steps) if st.spec is not None and st.spec.name.endswith(
            ("s1b2_expand", "s2b3_expand", "s3b5_expand"))]
        return s
    if kind == "convnext":
        s["x"] = _randn(g, case["batch"], case["image"], case["image"], 3)
        s["net"] = convnext.ConvNeXtStack(case["batch"], DEV, image=case["image"], seed=seed % 100000)
        last = tuple(f"s{i}b{d - 1}_pw2" for i, d in enumerate(convnext.DEPTHS[:-1]))
        s["taps"] = [i for i, st in enumerate(s["net"].steps) if st.name in last]
        return s
    if kind == "masks":
        s["layers"] = []
        for spec in synth.config_layers(5, 1):
            scale = case["width"] / 64.0
            cin, cout = int(spec.C_in * scale), int(spec.C_out * scale)
            desc = api.make_desc(1, spec.H, spec.W, cin, cout, spec.KH, spec.KW, stride=spec.stride, pad=spec.pad)
            w = _randn(g, cout, spec.KH, spec.KW, cin, std=1.0 / math.sqrt(spec.KH * spec.KW * cin))
            groups = w.numel() // 4
            s["layers"].append((desc, w, _randn(g, groups, 6, dtype=torch.float32), groups))
        return s
    desc = s["desc"] = _desc(case)
    ho, wo = _extent(case)
    k_in = case["cin"] // case.get("groups", 1)
    s["x"] = _randn(g, case["n"], case["h"], case["w"], case["cin"])
    s["bias"] = _randn(g, case["cout"], std=0.1, dtype=torch.float32)
    w = _randn(g, case["cout"], case["k"], case["k"], k_in, std=1.0 / math.sqrt(case["k"] ** 2 * k_in))
    s["w"] = w
    if kind == "train":
        n_groups = w.numel() // 4
        s["logits"], s["noise"] = _randn(g, n_groups, 6, dtype=torch.float32), _gumbel(g, n_groups, 6)
        s["dy"] = _randn(g, case["n"], ho, wo, case["cout"])
        s["m"], s["v"] = torch.zeros_like(s["logits"]), torch.zeros_like(s["logits"])
        s["step"] = 0
        return s
    if case["dtype"] == "e4m3":
        wq = api.ssconv_quantize_e4m3(w, W_SCALE)
        pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_E4M3, wq, w.numel() // 4)
        s["w_comp"], s["meta"] = api.ssconv_compress_fp8(desc, wq, pat)
        return s
    pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w, w.numel() // 4)
    if case["groups"] > 1:
        s["w_comp"], s["meta"] = api.ssconv_compress_grouped(desc, case["groups"], w, pat)
    else:
        s["w_comp"], s["meta"] = api.ssconv_compress(desc, w, pat)
    if case["res"]:
        s["residual"] = _randn(g, case["n"], ho, wo, case["cout"])
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("resnet", "convnext"):
        y = s["net"].forward(s["x"])
        return [s["net"].outputs[i] for i in s["taps"]] + [y]
    if kind == "masks":
        out = []
        for desc, w, scores, groups in s["layers"]:
            pattern = api.ssconv_select_mask(api.MASK_LOGITS_F32, scores, groups)
            out.append(api.ssconv_compress(desc, w, pattern))
        # (one tensor of values and one of metadata: the network's packed weights as a file holds them)
        return torch.cat([v for v, _ in out]), torch.cat([m for _, m in out])
    if kind == "layer":
        if case["dtype"] == "e4m3":
            xq = api.ssconv_quantize_e4m3(s["x"])
            return api.ssconv_forward_fp8(s["desc"], xq, s["w_comp"], s["meta"], s["bias"], 1.0 / W_SCALE)
        if case["groups"] > 1:
            return api.ssconv_forward_grouped(s["desc"], case["groups"], s["x"], s["w_comp"], s["meta"], s["bias"])
        return api.ssconv_forward(s["desc"], s["x"], s["w_comp"], s["meta"], s["bias"], residual=s.get("residual"))
    s["step"] += 1
    z, w_eff = api.ssconv_soft_mask(s["logits"], s["noise"], TAU, s["w"])
    y = api.ssconv_forward_dense(s["desc"], s["x"], w_eff, s["bias"])
    dw = api.ssconv_wgrad(s["desc"], s["x"], s["dy"])
    dx = api.ssconv_dgrad(s["desc"], s["dy"], w_eff)
    g_logits = api.ssconv_mask_grad(z, TAU, s["w"], dw)
    api.ssconv_adamw(s["logits"], g_logits, s["m"], s["v"], s["step"], lr=1e-3)
    return dict(y=y, dw=dw, dx=dx, g_logits=g_logits, logits=s["logits"], m=s["m"], v=s["v"])


# ----------------------------------------------------------------------------- what a pass cannot do without
def _conv_flops(positions, cout, k_total):
    return 2.0 * positions * cout * k_total


def work(case):
    """Bytes that have to cross memory once and floating-point operations.  A masked convolution multiplies the kept
    half of its weights; a network writes every step's output (its `outputs` hold them all after a pass)."""
    kind = case["kind"]
    if kind == "resnet":
        n = case["batch"]
        bytes_, flops = 2.0 * n * 224 * 224 * 3, 0.0
        for st in synth.resnet50_stack(n, residual=True):
            if st.kind == "maxpool":
                bytes_ += 2.0 * n * 56 * 56 * 64
                continue
            sp = st.spec
            masked = st.kind == "conv"
            cin = sp.C_in if masked else 3
            weights = sp.C_out * sp.KH * sp.KW * cin
            bytes_ += 2.0 * sp.P * sp.C_out + weights * (1.125 if masked else 2.0) + 4.0 * sp.C_out
            flops += _conv_flops(sp.P, sp.C_out, sp.KH * sp.KW * cin) * (0.5 if masked else 1.0)
        return dict(bytes=bytes_, flops=flops)
    if kind == "convnext":
        n, hw = case["batch"], case["image"] // 4
        bytes_ = 2.0 * n * case["image"] ** 2 * 3
        flops = _conv_flops(n * hw * hw, convnext.WIDTHS[0], 48)
        bytes_ += 2.0 * n * hw * hw * (48 + 2 * convnext.WIDTHS[0])
        prev = convnext.WIDTHS[0]
        for stage, (depth, c) in enumerate(zip(convnext.DEPTHS, convnext.WIDTHS)):
            if stage:
                bytes_ += 2.0 * n * hw * hw * prev                                 # layer norm before the downsampling
                hw //= 2
                flops += 0.5 * _conv_flops(n * hw * hw, c, 4 * prev)
                bytes_ += 2.0 * n * hw * hw * c + 1.125 * c * 4 * prev
                prev = c
            p = n * hw * hw
            flops += depth * (2.0 * p * c * 49 + 0.5 * _conv_flops(p, 4 * c, c) + 0.5 * _conv_flops(p, c, 4 * c))
            bytes_ += depth * (2.0 * p * (c + c + 4 * c + c) + 2.0 * 49 * c + 1.125 * 8 * c * c)
        return dict(bytes=bytes_, flops=flops)
    if kind == "masks":
        weights = sum(int(sp.C_in * case["width"] / 64.0) * int(sp.C_out * case["width"] / 64.0) * sp.KH * sp.KW
                      for sp in synth.config_layers(5, 1))
        return dict(bytes=weights * (24.0 / 4 + 2.0 + 1.125), flops=5.0 * weights / 4)   # scores and weights in, packed out
    ho, wo = _extent(case)
    p_out = case["n"] * ho * wo
    x = 2.0 * case["n"] * case["h"] * case["w"] * case["cin"]
    y = 2.0 * p_out * case["cout"]
    if kind == "layer":
        k_total = case["k"] ** 2 * case["cin"] // case["groups"]
        weights = case["cout"] * k_total * (1.125 if case["dtype"] == "bf16" else 0.5625)
        return dict(bytes=x + y * (2 if case["res"] else 1) + weights + 4.0 * case["cout"],
                    flops=0.5 * _conv_flops(p_out, case["cout"], k_total))
    k_total = case["k"] ** 2 * case["cin"]
    n_w = case["cout"] * k_total
    # x, dy, w, logits, noise, moments in; y, dx, dw, gradient of the choice weights, logits, moments out
    return dict(bytes=2 * x + 2 * y + n_w * (2.0 + 4.0 + 6.0 * 7), flops=3 * _conv_flops(p_out, case["cout"], k_total))


def tolerance(case):
    """Relative error that another correct implementation of the same precision shows (`max` in units of the result's
    root mean square, or of the value where that is larger): about four times what was measured.

    Layers and training steps, against the same arithmetic in 64 bits: 1.7e-3 and 4.7e-3 (one rounding to bf16), fp32
    results far below.  Networks, against the same chain of bf16 tensors with 32- or 64-bit sums, where single
    roundings fall the other way and are carried on: 4.0e-3 and 2.9e-2 (ResNet-50-shaped), 8.9e-3 and 3.6e-2
    (ConvNeXt-T-shaped)."""
    if case["kind"] == "masks":
        return "exact"
    if case["kind"] == "resnet":
        return dict(rel=1.6e-2, max=0.12)
    if case["kind"] == "convnext":
        return dict(rel=3.5e-2, max=0.15)
    return dict(rel=7e-3, max=2e-2)


# ----------------------------------------------------------------------------- the same in 64 bits, plain torch
_PAIRS = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))   # the positions the six patterns keep


def _keep_two(w):
    """w with the two largest magnitudes of each group of four kept (of equal ones the earlier), fp64."""
    v = w.double().reshape(-1, 4)
    a = v.abs()
    earlier = torch.ones(4, 4, dtype=torch.bool, device=v.device).tril(-1)                   # [i, j]: j before i
    beaten = (a[:, None, :] > a[:, :, None]) | ((a[:, None, :] == a[:, :, None]) & earlier)
    return torch.where(beaten.sum(2) < 2, v, torch.zeros_like(v)).reshape(w.shape)


def _patches(t, kh, kw, stride, ho, wo):
    return t[:, kh:kh + stride * (ho - 1) + 1:stride, kw:kw + stride * (wo - 1) + 1:stride]


def _conv(x, w, bias, stride=1, pad=0, act="none", res=None):
    """One matrix product per filter tap; x [N, H, W, C] and w [C_out, KH, KW, C]."""
    w = w.double()
    kh, kw = w.shape[1:3]
    xp = torch.nn.functional.pad(x, (0, 0, pad, pad, pad, pad)).double()
    ho, wo = (xp.shape[1] - kh) // stride + 1, (xp.shape[2] - kw) // stride + 1
    y = bias.double().expand(x.shape[0], ho, wo, w.shape[0]).clone()
    for i in range(kh):
        for j in range(kw):
            y += _patches(xp, i, j, stride, ho, wo) @ w[:, i, j].T
    if res is not None:
        y += res.double()
    return y.relu_() if act == "relu" else torch.nn.functional.gelu(y) if act == "gelu" else y


def _exact_layer(case, s, w):
    x, groups = s["x"], case["groups"]
    if case["dtype"] == "e4m3":
        x = x.float().clamp(-448, 448).to(torch.float8_e4m3fn).float()
        w = (w.float() * W_SCALE).clamp(-448, 448).to(torch.float8_e4m3fn).float()
    w = _keep_two(w)
    if case["dtype"] == "e4m3":
        w = w / W_SCALE
    y = [_conv(x_g, w_g, b_g, case["stride"], case["pad"], case["act"], s.get("residual")) for x_g, w_g, b_g in
         zip(x.chunk(groups, 3), w.chunk(groups, 0), s["bias"].chunk(groups))]
    return torch.cat(y, 3)


def _exact_train(case, s):
    k, st, pad = case["k"], case["stride"], case["pad"]
    ho, wo = _extent(case)
    d = torch.zeros(4, 6, dtype=torch.float64, device=DEV)
    for i, kept in enumerate(_PAIRS):
        d[list(kept), i] = 1.0
    w, dy = s["w"].double(), s["dy"].double()
    z = torch.softmax((s["logits"].double() + s["noise"].double()) / TAU, 1)
    # (the effective weights are a bf16 tensor between two calls)
    w_eff = ((z @ d.T) * w.reshape(-1, 4)).reshape(w.shape).to(torch.bfloat16).double()
    xp = torch.nn.functional.pad(s["x"], (0, 0, pad, pad, pad, pad)).double()
    dw, dxp = torch.zeros_like(w), torch.zeros_like(xp)
    for i in range(k):
        for j in range(k):
            dw[:, i, j] = dy.reshape(-1, case["cout"]).T @ _patches(xp, i, j, st, ho, wo).reshape(-1, case["cin"])
            _patches(dxp, i, j, st, ho, wo).add_(dy @ w_eff[:, i, j])
    g_z = (dw.reshape(-1, 4) * w.reshape(-1, 4)) @ d
    g = z * (g_z - (z * g_z).sum(1, keepdim=True)) / TAU
    m, v = 0.1 * g, 0.001 * g * g                                 # the first step, from zero moments
    theta = s["logits"].double()
    theta = theta - 1e-3 * (m / 0.1 / ((v / 0.001).sqrt() + 1e-8) + 1e-4 * theta)
    return dict(y=_conv(s["x"], w_eff, s["bias"], st, pad), dw=dw, dx=dxp[:, pad:pad + case["h"], pad:pad + case["w"]],
                g_logits=g, logits=theta, m=m, v=v)


def _exact_resnet(s):
    net, outs = s["net"], []
    last = {}                                                     # the step that reads an output last
    for i, st in enumerate(net.steps):
        last[st.src] = last[st.res] = i
    for i, st in enumerate(net.steps):
        x = s["x"] if st.src < 0 else outs[st.src]
        if st.kind == "maxpool":
            y = torch.nn.functional.max_pool2d(x.permute(0, 3, 1, 2), 3, 2, 1).permute(0, 2, 3, 1)
        else:
            sp = st.spec
            inp = synth.make_weights(sp)
            w = inp.w.to(DEV)
            w = _keep_two(w) if st.kind == "conv" else w[..., :x.shape[3]]
            y = _conv(x, w, inp.bias.to(DEV), sp.stride, sp.pad, "relu" if sp.relu else "none",
                      outs[st.res] if st.res >= 0 else None)
        outs.append(y)
        for k in range(i):
            if k not in s["taps"] and last.get(k, 0) <= i:
                outs[k] = None
    return [outs[i] for i in s["taps"]] + [outs[-1]]


def _exact_convnext(s):
    net, outs = s["net"], []
    for i, (st, p) in enumerate(zip(net.steps, net.params)):
        x = s["x"] if st.src < 0 else outs[st.src]
        if st.kind == "s2d":
            y = x                                                 # the dense stem below reads the image itself
        elif st.kind == "dense":
            y = _conv(x, p["w_host"].to(DEV), p["bias"], 4)
        elif st.kind == "layernorm":
            y = torch.nn.functional.layer_norm(x.double(), x.shape[3:], p["gamma"].double(), p["beta"].double(), convnext.LN_EPS)
        elif st.kind == "depthwise":
            xp = torch.nn.functional.pad(x, (0, 0, 3, 3, 3, 3))
            y = p["bias"].double().expand(x.shape).clone()
            for a in range(7):
                for b in range(7):
                    y += _patches(xp, a, b, 1, *x.shape[1:3]) * p["w"][a, b].double()
        else:
            y = _conv(x, _keep_two(p["w_host"].to(DEV)), p["bias"], st.desc.stride_h, 0, "gelu" if st.gelu else "none",
                      outs[st.res] if st.res >= 0 else None)
        outs.append(y)
        for k in range(max(0, i - 3)):                            # a block's input is read at most four steps later
            if k not in s["taps"]:
                outs[k] = None
    return [outs[i] for i in s["taps"]] + [outs[-1]]


def exact(case, seed):
    """What `run` returns for these inputs, in 64 bits and by plain torch operations.  A network is one chain in
    64 bits, without the rounding of the tensors in between."""
    if case["kind"] == "masks":
        return None                                               # bytes
    s = prepare(case, seed)
    if case["kind"] == "resnet":
        return _exact_resnet(s)
    if case["kind"] == "convnext":
        return _exact_convnext(s)
    if case["kind"] == "train":
        return _exact_train(case, s)
    return _exact_layer(case, s, s["w"])
