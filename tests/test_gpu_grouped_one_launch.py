"""All channel groups in one launch: against one launch per group on the same slices (bit for bit where both walk whole
tiles of the same width order, so within the oracle's tolerance in general), at group widths on both sides of the
rule, ragged output channels and several channel tiles per group; and infinities stay in their group."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import blocks, masks
from oracle.conv import ConvShape
from paper_2411_00288_b200 import api, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [  # N, H, W, C_in per group, C_out per group, K, stride, pad, groups, sparse, act, one launch
    (3, 14, 14, 32, 72, 3, 1, 1, 3, True, "relu", True),
    (2, 15, 11, 64, 136, 3, 2, 1, 2, True, "none", True),     # two channel tiles, the second nearly empty
    (4, 28, 28, 96, 264, 1, 1, 0, 4, True, "gelu", True),     # three channel tiles, half-filled last k-block
    (2, 9, 9, 16, 40, 3, 1, 1, 4, True, "relu", False),       # an MMA would reach into the next group
    (2, 9, 9, 40, 48, 3, 1, 1, 3, True, "relu", False),
    (3, 14, 14, 16, 72, 3, 1, 1, 3, False, "relu", True),
    (7, 30, 28, 80, 200, 3, 1, 1, 2, False, "gelu", True),
    (2, 9, 9, 24, 48, 3, 1, 1, 3, False, "relu", False),
    # a full k-block followed by one that is partly the group's own
    (4, 28, 28, 96, 264, 1, 1, 0, 4, True, "relu", True),
    (7, 30, 28, 80, 200, 3, 1, 1, 2, False, "none", True),
]


def _run(case, x, w, bias):
    N, H, W, ci, co, K, s, p, groups, sparse, act, _ = case
    desc = api.make_desc(N, H, W, groups * ci, groups * co, K, K, s, p, bias=True, relu=act == "relu", gelu=act == "gelu")
    if not sparse:
        c0 = api.ssconv_launch_count()
        return api.ssconv_forward_dense_grouped(desc, groups, x, w, bias), api.ssconv_launch_count() - c0
    pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w, w.numel() // 4)
    comp = api.ssconv_compress_grouped(desc, groups, w, pat)
    c0 = api.ssconv_launch_count()
    return api.ssconv_forward_grouped(desc, groups, x, *comp, bias), api.ssconv_launch_count() - c0


def _inputs(case):
    N, H, W, ci, co, K, s, p, groups, sparse, act, _ = case
    g = torch.Generator().manual_seed(synth.SEED_BASE + 7500 + CASES.index(case))
    x = torch.randn((N, H, W, groups * ci), generator=g).to(torch.bfloat16)
    w = (torch.randn((groups * co, K, K, ci), generator=g) / (K * K * ci) ** 0.5).to(torch.bfloat16)
    return x, w, torch.randn((groups * co,), generator=g) * 0.1


@pytest.mark.parametrize("case", CASES, ids=[f"{c[3]}to{c[4]}_g{c[8]}_{'sparse' if c[9] else 'dense'}_{c[10]}" for c in CASES])
def test_groups_in_one_launch_match_oracle(case):
    N, H, W, ci, co, K, s, p, groups, sparse, act, one = case
    x, w, bias = _inputs(case)
    y, launches = _run(case, x.to(DEV), w.to(DEV), bias.to(DEV))
    torch.cuda.synchronize()
    assert (launches == 1) == one
    shape = ConvShape(N, H, W, groups * ci, groups * co, K, K, (s, s), (p, p), (1, 1), relu=False)
    mask = masks.mask_from_pattern(masks.select_from_magnitude(synth.bf16_bits(w)), tuple(w.shape)) if sparse else None
    ref = blocks.grouped_conv2d_f64(shape, groups, synth.bf16_bits(x), synth.bf16_bits(w), mask=mask, bias=bias.numpy())
    ref = parity.gelu_f64(ref) if act == "gelu" else np.maximum(ref, 0.0) if act == "relu" else ref
    rel, mx = parity.errors(parity.bf16_tensor_to_f64(y), ref)
    assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, (rel, mx)


@pytest.mark.parametrize("case", [c for c in CASES if c[10] != "gelu"], ids=[f"{c[3]}to{c[4]}_g{c[8]}_{'sparse' if c[9] else 'dense'}" for c in CASES if c[10] != "gelu"])
def test_an_infinite_pixel_stays_in_its_group(case):
    N, H, W, ci, co, K, s, p, groups, sparse, act, _ = case
    x, w, bias = _inputs(case)
    clean, _ = _run(case, x.to(DEV), w.to(DEV), bias.to(DEV))
    x[0, 4, 4, ci:2 * ci] = float("inf")                           # the second group's channels at one pixel
    y, _ = _run(case, x.to(DEV), w.to(DEV), bias.to(DEV))
    assert torch.equal(y[..., :co], clean[..., :co]) and torch.equal(y[..., 2 * co:], clean[..., 2 * co:])
    assert not bool(torch.isfinite(y[..., co:2 * co].float()).all())


PLANS = [  # N, H, C_in, C_out, groups, K, act, workspace, launches (2:4)
    (32, 56, 192, 768, 2, 1, "gelu", True, 2),        # paced by the epilogue: two sets of epilogue groups in each launch
    (32, 56, 192, 768, 2, 1, "relu", True, 1),
    (16, 28, 128, 256, 2, 1, "gelu", True, 1),        # too few tiles to make up for a launch
    (1, 7, 2048, 2048, 2, 3, "none", True, 4),        # K split in each launch, and a finishing kernel
    (1, 7, 2048, 2048, 2, 3, "none", False, 1),       # no scratch, no split: all groups' tiles together
]


@pytest.mark.parametrize("plan", PLANS, ids=[f"{p[0]}x{p[1]}_{p[2]}to{p[3]}_g{p[4]}_{p[6]}_{'ws' if p[7] else 'no_ws'}" for p in PLANS])
def test_launches_of_a_grouped_layer(plan):
    N, H, ci, co, groups, K, act, with_ws, launches = plan
    g = torch.Generator(device=DEV).manual_seed(synth.SEED_BASE + 7600)
    x = torch.randn((N, H, H, ci), generator=g, device=DEV).to(torch.bfloat16)
    w = (torch.randn((co, K, K, ci // groups), generator=g, device=DEV) / (K * K * ci / groups) ** 0.5).to(torch.bfloat16)
    desc = api.make_desc(N, H, H, ci, co, K, K, 1, K // 2, bias=False, relu=act == "relu", gelu=act == "gelu")
    pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w, w.numel() // 4)
    w_comp, meta = api.ssconv_compress_grouped(desc, groups, w, pat)
    y = torch.empty((N, H, H, co), dtype=torch.bfloat16, device=DEV)
    ws = api.default_workspace(x.device)
    c0 = api.ssconv_launch_count()
    rc = api.lib().ssconv_forward_grouped(ctypes.byref(desc), groups, x.data_ptr(), w_comp.data_ptr(), meta.data_ptr(), None, y.data_ptr(),
                                          ws.data_ptr() if with_ws else None, ws.numel() if with_ws else 0, None, None)
    assert rc == api.OK and api.ssconv_launch_count() - c0 == launches
    torch.cuda.synchronize()
    # each group as a layer of its own on a copy of its channels
    ci_g, co_g = ci // groups, co // groups
    one = api.make_desc(N, H, H, ci_g, co_g, K, K, 1, K // 2, bias=False, relu=act == "relu", gelu=act == "gelu")
    for i in range(groups):
        wi = w[i * co_g:(i + 1) * co_g].contiguous()
        comp = api.ssconv_compress(one, wi, api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, wi, wi.numel() // 4))
        ref = api.ssconv_forward(one, x[..., i * ci_g:(i + 1) * ci_g].contiguous(), *comp).float()
        err = (y[..., i * co_g:(i + 1) * co_g].float() - ref).abs()
        assert bool((err <= 2.0 ** -7 * ref.abs() + 1e-3).all())   # (K split or not: another order of summation)
