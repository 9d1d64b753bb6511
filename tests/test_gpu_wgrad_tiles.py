"""Weight gradient of pointwise layers whose work items hold several tiles of output channels."""
import pytest
import torch

from paper_2411_00288_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# n, h, w, c_in, c_out: enough positions for long ranges on every SM
CASES = [
    ("three_tiles",   64, 56, 56, 96,  384),
    ("ragged_two",    64, 56, 56, 40,  200),      # channels no multiple of 64: two copies per tile
    ("five_tiles",    32, 64, 64, 128, 520),      # items of three and of two tiles, the last with 8 channels
    ("one_k_block",   48, 56, 56, 64,  256),
    ("one_tile",      60, 56, 57, 72,  72),       # one tile, on a deeper ring
    ("few_slices",    2,  16, 17, 24,  136),      # fewer slices than sets of adding threads, K no multiple of 8 x 3
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_wgrad_items_of_several_channel_tiles(case):
    name, n, h, w, ci, co = case
    g = torch.Generator(device=DEV).manual_seed(7100 + CASES.index(case))
    desc = api.make_desc(n, h, w, ci, co, 1, 1, bias=False)
    x = torch.randn((n, h, w, ci), generator=g, device=DEV).to(torch.bfloat16)
    dy = torch.randn((n, h, w, co), generator=g, device=DEV).to(torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    dw = api.ssconv_wgrad(desc, x, dy, dev_status=status)
    again = api.ssconv_wgrad(desc, x, dy)
    ref = dy.reshape(-1, co).double().T @ x.reshape(-1, ci).double()
    rel = float((dw.reshape(co, ci).double() - ref).norm() / ref.norm())
    assert int(status.item()) == 0
    assert rel <= 1e-4, f"{name}: {rel:.3e}"      # fp32 sums of exact products, as for every weight gradient
    assert torch.equal(dw, again)


@pytest.mark.parametrize("case", CASES[:3], ids=[c[0] for c in CASES[:3]])
def test_wgrad_in_the_scratch_of_items_of_one_channel_tile(case):
    name, n, h, w, ci, co = case
    n *= 2                                                      # (enough positions for items of several tiles)
    g = torch.Generator(device=DEV).manual_seed(7150 + CASES.index(case))
    desc = api.make_desc(n, h, w, ci, co, 1, 1, bias=False)
    x = torch.randn((n, h, w, ci), generator=g, device=DEV).to(torch.bfloat16)
    dy = torch.randn((n, h, w, co), generator=g, device=DEV).to(torch.bfloat16)
    tiles, steps = -(-co // 128), -(-n * h * w // 64)
    ranges = torch.cuda.get_device_properties(0).multi_processor_count // tiles
    ranges = -(-steps // -(-steps // ranges))                   # (none of them empty)
    small = ranges * tiles * 128 * ci * 4
    need = api.ssconv_wgrad_ws_bytes(desc)
    assert small < need
    ws = torch.empty(need, dtype=torch.uint8, device=DEV)
    ref = dy.reshape(-1, co).double().T @ x.reshape(-1, ci).double()
    for size in (small, need - 16, need):
        dw = api.ssconv_wgrad(desc, x, dy, ws=ws[:size])
        assert float((dw.reshape(co, ci).double() - ref).norm() / ref.norm()) <= 1e-4, size
    with pytest.raises(api.SsconvError):
        api.ssconv_wgrad(desc, x, dy, ws=ws[:small - 16])
