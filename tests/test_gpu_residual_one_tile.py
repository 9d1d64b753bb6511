"""Residual layers whose thread blocks have one tile at most: an epilogue of their own (all residual pieces brought in at the
start, the stores issued by the epilogue).  Against the oracle around the line (as many tiles as SMs, one row of tiles more),
at every staged width, with ragged channels and short last tiles, and in place."""
import pytest
import torch

from paper_2411_00288_b200 import api, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

LAYERS = [  # N, H, W, C_in, C_out, k, pad, relu, gelu
    (1, 14, 14, 64, 64, 3, 1, True, False),
    (1, 9, 11, 64, 136, 1, 0, False, False),       # a channel tile of eight
    (3, 23, 19, 40, 264, 3, 1, False, True),
    (1, 148, 160, 32, 128, 1, 0, True, False),     # 148 tiles of 160 positions
    (1, 149, 160, 32, 128, 1, 0, True, False),     # 149: a block with two
]


@pytest.mark.parametrize("sparse", [True, False], ids=["sparse", "dense"])
@pytest.mark.parametrize("width", [0, 48, 80, 112, 160])
@pytest.mark.parametrize("layer", LAYERS, ids=["x".join(map(str, v[:5])) for v in LAYERS])
def test_residual_with_one_tile_per_block(layer, width, sparse):
    N, H, W, ci, co, k, pad, relu, gelu = layer
    spec = synth.LayerSpec("res1", N, H, W, ci, co, k, k, 1, pad, 1, relu=relu, gelu=gelu, w_std="fan_in", mask_source="magnitude",
                           config=8, index=400 + LAYERS.index(layer))
    api.ssconv_tune(api.TUNE_TILE_POSITIONS, width)
    try:
        rel, mx = parity.check_layer(spec, DEV, sparse=sparse, sample=20000, residual=True)
    finally:
        api.ssconv_tune(api.TUNE_TILE_POSITIONS, 0)
    assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, (rel, mx)


def test_in_place_and_repeated():
    g = torch.Generator(device=DEV).manual_seed(synth.SEED_BASE + 7700)
    x = torch.randn((2, 28, 28, 128), generator=g, device=DEV).to(torch.bfloat16)
    w = (torch.randn((200, 1, 1, 128), generator=g, device=DEV) / 11).to(torch.bfloat16)
    res = torch.randn((2, 28, 28, 200), generator=g, device=DEV).to(torch.bfloat16)
    desc = api.make_desc(2, 28, 28, 128, 200, 1, 1, bias=False)
    comp = api.ssconv_compress(desc, w, api.ssconv_select_mask(api.MASK_MAGNITUDE_BF16, w, w.numel() // 4))
    ref = api.ssconv_forward(desc, x, *comp, residual=res)
    for _ in range(50):   # back to back: the set-up of each launch overlaps the one before
        y = res.clone()
        api.ssconv_forward(desc, x, *comp, y=y, residual=y)
        assert torch.equal(y, ref)
