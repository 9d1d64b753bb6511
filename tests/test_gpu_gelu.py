"""The GELU epilogue: its values over every bf16 number, and the form with two sets of epilogue groups at the edges of
its tiles (odd numbers of tiles, a short last tile, ragged channels, every staged width, slices of a wider tensor)."""
import math

import numpy as np
import pytest
import torch

from oracle import blocks, masks
from oracle.conv import ConvShape
from paper_2411_00288_b200 import api, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_gelu_of_every_bf16_value():
    bits = torch.arange(0, 65536, dtype=torch.int32).to(torch.uint16)
    v = bits.view(torch.bfloat16)
    v = v[~(torch.isfinite(v) & (v.abs() > 1e30))]            # (x 0.5 x stays finite)
    pad = (-v.numel()) % 64
    v = torch.cat([v, torch.zeros(pad, dtype=torch.bfloat16)])
    x = torch.zeros((1, v.numel() // 64, 64, 16), dtype=torch.bfloat16)
    x[0, :, :, 0] = v.view(-1, 64)
    w = torch.zeros((16, 1, 1, 16), dtype=torch.bfloat16)
    w[:, 0, 0, 0] = 1.0
    desc = api.make_desc(1, x.shape[1], 64, 16, 16, 1, 1, bias=False, gelu=True)
    pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w.to(DEV), w.numel() // 4)
    comp = api.ssconv_compress(desc, w.to(DEV), pat)
    y = api.ssconv_forward(desc, x.to(DEV), *comp).cpu()
    for c in (0, 7, 15):
        got = y[0, :, :, c].reshape(-1)
        nan = torch.isnan(v)
        assert bool(torch.isnan(got[nan]).all())
        assert bool((got[v == float("inf")] == float("inf")).all())
        fin = torch.isfinite(v)
        ref = parity.gelu_f64(v[fin].double().numpy())
        err = np.abs(got[fin].double().numpy() - ref)
        # one rounding to bf16 (half a unit in the last of 8 bits: at most 2^-8 of the value), 3.3e-5 of the fp32
        # evaluation, and the clamp's 2e-8 x 5.7 far below zero
        assert (err <= (2.0 ** -8 + 5e-5) * np.abs(ref) + 2e-7).all(), float((err - 2.0 ** -8 * np.abs(ref)).max())


def test_gelu_far_below_zero_and_at_minus_infinity():
    bits = torch.arange(0x8000, 0x10000, dtype=torch.int32).to(torch.uint16)       # every bf16 number below zero
    v = bits.view(torch.bfloat16)
    x = torch.zeros((1, v.numel() // 64, 64, 16), dtype=torch.bfloat16)
    x[0, :, :, 0] = v.view(-1, 64)
    w = torch.zeros((16, 1, 1, 16), dtype=torch.bfloat16)
    w[:, 0, 0, 0] = 1.0
    desc = api.make_desc(1, x.shape[1], 64, 16, 16, 1, 1, bias=False, gelu=True)
    pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w.to(DEV), w.numel() // 4)
    comp = api.ssconv_compress(desc, w.to(DEV), pat)
    got = api.ssconv_forward(desc, x.to(DEV), *comp).cpu()[0, :, :, 5].reshape(-1)
    assert bool(torch.isnan(got[v == float("-inf")]).all())                        # as x Phi(x) in fp64
    fin = torch.isfinite(v)
    z = v[fin].double().numpy()
    ref = z * 0.5 * np.vectorize(math.erfc)(-z / math.sqrt(2.0))                   # (no cancellation below zero)
    err = np.abs(got[fin].double().numpy() - ref)
    # one rounding to bf16 (half a unit in the last of 8 bits), the evaluation's 5.1e-6, and 6.1e-13 below -5.54, where the
    # polynomial is not fitted
    assert (err <= (2.0 ** -8 + 1e-5) * np.abs(ref) + 1e-12).all(), float((err - 2.0 ** -8 * np.abs(ref)).max())


LAYERS = [  # N, H, W, C_in, C_out, k, pad
    (16, 56, 56, 96, 384, 1, 0),
    (1, 160, 150, 16, 128, 1, 0),      # about one tile per thread block and a few with two
    (3, 97, 83, 40, 136, 1, 0),        # ragged channels, an odd number of tiles, a short last one
    (5, 57, 41, 64, 72, 1, 0),         # half a channel tile
    (2, 120, 117, 24, 256, 2, 1),      # four taps
]


@pytest.mark.parametrize("layer", LAYERS, ids=["x".join(map(str, v[:5])) for v in LAYERS])
@pytest.mark.parametrize("width", [0, 48, 112, 160, 208])
def test_two_epilogue_sets_match_oracle(layer, width):
    N, H, W, ci, co, k, pad = layer
    spec = synth.LayerSpec("gelu2", N, H, W, ci, co, k, k, 1, pad, 1, gelu=True, w_std="fan_in", mask_source="magnitude",
                           config=8, index=300 + LAYERS.index(layer))
    api.ssconv_tune(api.TUNE_TILE_POSITIONS, width)
    try:
        for sparse in (True, False):
            rel, mx = parity.check_layer(spec, DEV, sparse=sparse, sample=20000)
            assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, (sparse, rel, mx)
    finally:
        api.ssconv_tune(api.TUNE_TILE_POSITIONS, 0)


@pytest.mark.parametrize("sparse,ci_g,co_g", [(False, 32, 144), (False, 24, 144), (True, 40, 136)], ids=["one_launch", "dense", "sparse"])
def test_two_epilogue_sets_on_channel_slices(sparse, ci_g, co_g):
    # 24 and 40 channels per group: the last MMA would reach into the next group, so that every group is a launch of its own, on
    # strided views and with two sets of epilogue groups (350 tiles); 32 dense ones go in one launch with one set
    N, H, W, groups = 4, 90, 77, 2
    ci, co = groups * ci_g, groups * co_g
    g = torch.Generator().manual_seed(synth.SEED_BASE + 7300)
    x = torch.randn((N, H, W, ci), generator=g).to(torch.bfloat16)
    w = (torch.randn((co, 1, 1, ci_g), generator=g) / ci_g ** 0.5).to(torch.bfloat16)
    bias = torch.randn((co,), generator=g) * 0.1
    desc = api.make_desc(N, H, W, ci, co, 1, 1, bias=True, gelu=True)
    mask = None
    if sparse:
        pat = api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w.to(DEV), w.numel() // 4)
        comp = api.ssconv_compress_grouped(desc, groups, w.to(DEV), pat)
        mask = masks.mask_from_pattern(masks.select_from_magnitude(synth.bf16_bits(w)), tuple(w.shape))
    c0 = api.ssconv_launch_count()
    y = (api.ssconv_forward_grouped(desc, groups, x.to(DEV), *comp, bias.to(DEV)) if sparse else
         api.ssconv_forward_dense_grouped(desc, groups, x.to(DEV), w.to(DEV), bias.to(DEV)))
    assert api.ssconv_launch_count() - c0 == (1 if ci_g == 32 else groups)
    torch.cuda.synchronize()
    shape = ConvShape(N, H, W, ci, co, 1, 1, (1, 1), (0, 0), (1, 1), relu=False)
    ref = parity.gelu_f64(blocks.grouped_conv2d_f64(shape, groups, synth.bf16_bits(x), synth.bf16_bits(w), mask=mask, bias=bias.numpy()))
    rel, mx = parity.errors(parity.bf16_tensor_to_f64(y), ref)
    assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, (rel, mx)
