"""GPU parity of the kernel whose CTAs of a cluster share a tile's K, forced to 2, 4 and 8 of them."""
import pytest
import torch

from paper_2411_00288_b200 import api, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# name, n, h, w, c_in, c_out, k, stride, pad, activation, residual, tile width
CASES = [
    ("shares_of_one_group",  1, 7,  7,  1024, 128, 1, 1, 0, "relu", False, 64),   # 8 groups on 8 CTAs
    ("uneven_shares",        1, 7,  7,  576,  64,  3, 1, 1, "none", True,  64),   # 81 k-blocks: a last group of one
    ("channel_tail",         1, 9,  9,  200,  72,  3, 1, 1, "gelu", True,  48),   # a chunk of 8 channels, 72 of 128 rows
    ("two_channel_tiles",    2, 7,  7,  512,  264, 3, 1, 1, "relu", False, 64),   # the third tile has 8 channels
    ("positions_cut_short",  1, 9,  5,  1024, 96,  1, 1, 0, "gelu", False, 240),  # 45 positions: blocks past the last one
    ("one_position",         1, 1,  1,  2048, 128, 1, 1, 0, "none", False, 48),
    ("strided_two_images",   2, 15, 13, 128,  128, 3, 2, 1, "relu", True,  80),
]


@pytest.fixture
def tune():
    yield api.ssconv_tune
    api.ssconv_tune(api.TUNE_CLUSTER, -1)
    api.ssconv_tune(api.TUNE_TILE_POSITIONS, 0)


@pytest.mark.parametrize("size", [2, 4, 8])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_shared_k_matches_the_oracle(case, size, tune):
    name, n, h, w, ci, co, k, s, p, act, res, width = case
    spec = synth.LayerSpec(name, n, h, w, ci, co, k, k, s, p, 1, relu=act == "relu", gelu=act == "gelu", w_std="fan_in",
                           mask_source="magnitude", config=8, index=300 + CASES.index(case))
    desc = api.desc_from_spec(spec)
    for sparse in (True, False):
        tune(api.TUNE_CLUSTER, size)
        tune(api.TUNE_TILE_POSITIONS, width)
        plan = api.ssconv_plan(desc, sparse)
        tiles = -(-spec.P // width) * -(-co // 128)
        assert plan["split"] and plan["tile_positions"] == width and plan["ctas"] == tiles * size, plan
        rel, mx = parity.check_layer(spec, DEV, sparse=sparse, residual=res)
        # (the order of an fp32 sum is all that sets it apart from whole tiles: the gates are the layer's own)
        assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, f"{name} {sparse}: rel={rel:.3e} max={mx:.3e}"


def test_one_launch_no_scratch_and_the_same_bits_again():
    spec = synth.LayerSpec("again", 1, 14, 14, 256, 256, 3, 3, 1, 1, 1, relu=True, w_std="fan_in", mask_source="magnitude",
                           config=8, index=320)
    inp = synth.make_inputs(spec)
    desc = api.desc_from_spec(spec)
    w = inp.w.to(DEV)
    w_comp, meta = api.ssconv_compress(desc, w, parity.gpu_pattern(inp, DEV))
    ws = torch.full((api.ssconv_sizes(desc).ws_bytes_sparse,), 0x5A, dtype=torch.uint8, device=DEV)
    x, b = inp.x.to(DEV), inp.bias.to(DEV)
    n0 = api.ssconv_launch_count()
    y1 = api.ssconv_forward(desc, x, w_comp, meta, b, ws=ws)
    assert api.ssconv_launch_count() - n0 == 1
    y2 = api.ssconv_forward(desc, x, w_comp, meta, b, ws=ws[:16])   # (a scratch too small to split over the grid)
    torch.cuda.synchronize()
    assert torch.equal(y1, y2) and bool((ws == 0x5A).all())
