"""The 7 x 7 depthwise kernel on tensor cores at the sizes where its tiling can go wrong, against the fp64 oracle:
groups of sixteen windows that end inside an image, span several or are mostly empty, map widths around multiples
of eight, paddings up to the filter's width, one output row, more blocks' ranges than rows; and infinities and
NaNs, which may only reach the outputs whose own window holds them."""
import numpy as np
import pytest
import torch

from oracle import blocks
from oracle.conv import ConvShape
from paper_2411_00288_b200 import api, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture
def no_small_maps():
    """Small maps on the tensor-core kernel, as larger ones are."""
    api.ssconv_tune(api.TUNE_DEPTHWISE_SMALL, 0)
    yield
    api.ssconv_tune(api.TUNE_DEPTHWISE_SMALL, -1)


@pytest.fixture(params=[0, -1], ids=["tensor_cores", "small_maps"])
def either_kernel(request):
    """Small maps on the tensor-core kernel, whose bands meet pixels outside an output's window, and on their own."""
    api.ssconv_tune(api.TUNE_DEPTHWISE_SMALL, request.param)
    yield
    api.ssconv_tune(api.TUNE_DEPTHWISE_SMALL, -1)


CASES = [  # N, H, W, C, pad, relu
    (1, 7, 7, 32, 0, False),      # one output
    (1, 1, 1, 32, 3, True),       # one pixel
    (15, 9, 8, 32, 3, False),     # 15 windows
    (16, 9, 8, 64, 3, True),      # 16
    (17, 9, 8, 32, 3, False),     # 17: a second, nearly empty group
    (3, 30, 57, 96, 3, False),    # 8 windows per row, one column in the last
    (2, 12, 130, 32, 6, True),    # a row longer than a group of windows, padding of a whole filter
    (5, 8, 23, 160, 2, False),
    (40, 15, 15, 32, 4, False),   # block ranges that start and end inside a strip
]
CASES += [
    (12, 14, 14, 384, 3, True),   # units of rows cut into runs of two and three
    (9, 27, 30, 160, 3, False),   # (15 units of 27 rows: nine runs of three)
    (17, 9, 8, 2560, 3, False),   # 160 units of nine rows: ranges that cross from one into the next
    (96, 5, 7, 256, 3, False),    # 48 units of five rows: runs of one and two
    (3, 7, 21, 32, 3, True),      # (the fp32 kernel's tiles of 7 columns)
    (4, 4, 4, 608, 3, False),     # 64 pixels and 76 runs of rows, and on the other sides of that line
    (5, 4, 4, 608, 3, True),
    (4, 4, 4, 576, 3, False),
    (1, 5, 12, 96, 3, True),
    (30, 3, 8, 64, 3, False),     # three rows of one window, and on the other sides of that line
    (30, 3, 9, 64, 3, False),
    (30, 4, 8, 64, 3, True),
]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:4])) + f"_p{c[4]}" for c in CASES])
def test_depthwise7_at_the_edges_of_its_tiles(case):
    _check_case(case)


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:4])) + f"_p{c[4]}" for c in CASES])
def test_depthwise7_on_the_fp32_kernels(case):
    # where the tensor-core kernel is not run (another register count than its roles' split needs, maps too small)
    api.ssconv_tune(api.TUNE_DEPTHWISE_MMA, 0)
    try:
        _check_case(case)
    finally:
        api.ssconv_tune(api.TUNE_DEPTHWISE_MMA, -1)


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:4])) + f"_p{c[4]}" for c in CASES])
def test_depthwise7_without_the_kernel_for_small_maps(case, no_small_maps):
    # (most of the maps above are small: the tensor-core kernel at the edges of its own tiles)
    _check_case(case)


SMALL_CASES = [
    (1, 4, 8, 32, 3, False),      # one tile exactly
    (2, 5, 9, 64, 3, True),       # one row and one column more
    (1, 10, 14, 32, 0, False),    # no padding: the tile's pixels are the map
    (3, 3, 23, 96, 5, False),     # wide padding, rows of three tiles
    (2, 1, 1, 960, 6, True),      # many channels, windows mostly outside
    (37, 14, 14, 160, 3, False),  # 1480 blocks: the most
    (38, 14, 14, 160, 3, False),  # (one image more: the tensor-core kernel)
]


@pytest.mark.parametrize("case", SMALL_CASES, ids=lambda c: "x".join(map(str, c[:4])) + f"_p{c[4]}")
def test_depthwise7_on_small_maps(case):
    _check_case(case)


def _check_case(case):
    N, H, W, C, pad, relu = case
    g = torch.Generator().manual_seed(synth.SEED_BASE + 7100 + (CASES + SMALL_CASES).index(case))
    x = torch.randn((N, H, W, C), generator=g).to(torch.bfloat16)
    w = (torch.randn((7, 7, C), generator=g) / 7).to(torch.bfloat16)
    bias = torch.randn((C,), generator=g) * 0.1
    desc = api.make_desc(N, H, W, C, C, 7, 7, 1, pad, bias=True, relu=relu)
    Ho, Wo = api.ssconv_out_shape(desc)
    band = 256
    buf = torch.full((N * Ho * Wo * C + 2 * band,), -5.0, dtype=torch.bfloat16, device=DEV)
    y = buf[band:band + N * Ho * Wo * C].view(N, Ho, Wo, C)
    api.ssconv_depthwise(desc, x.to(DEV), w.to(DEV), bias.to(DEV), y=y)
    torch.cuda.synchronize()
    assert bool((buf[:band] == -5.0).all()) and bool((buf[-band:] == -5.0).all())
    shape = ConvShape(N, H, W, C, C, 7, 7, (1, 1), (pad, pad), (1, 1), relu=False)
    ref = blocks.depthwise_conv2d_f64(shape, synth.bf16_bits(x), synth.bf16_bits(w), bias=bias.numpy())
    if relu:
        ref = np.maximum(ref, 0.0)
    rel, mx = parity.errors(parity.bf16_tensor_to_f64(y), ref)
    assert rel <= parity.REL_FRO_TOL and mx <= parity.MAX_ABS_TOL, (case, rel, mx)


@pytest.mark.parametrize("polls", [0, 1, 3, 40])
@pytest.mark.parametrize("case", [(17, 9, 8, 2560, 3, False), (24, 28, 28, 64, 3, True), (9, 27, 30, 160, 3, False)])
def test_depthwise7_computes_everything_again_when_waits_run_out(case, polls, no_small_maps):
    # (0: all waits give up; more: some warps of a block may give up and others not)
    N, H, W, C, pad, relu = case
    g = torch.Generator(device=DEV).manual_seed(synth.SEED_BASE + 7990)
    x = torch.randn((N, H, W, C), generator=g, device=DEV).to(torch.bfloat16)
    w = (torch.randn((7, 7, C), generator=g, device=DEV) / 7).to(torch.bfloat16)
    bias = torch.randn(C, generator=g, device=DEV) * 0.1
    desc = api.make_desc(N, H, W, C, C, 7, 7, 1, pad, bias=True, relu=relu)
    ref = api.ssconv_depthwise(desc, x, w, bias)                                   # (compared with the oracle above)
    y = api.ssconv_selftest_depthwise_give_up(desc, x, w, bias, polls)
    again = api.ssconv_depthwise(desc, x, w, bias)
    torch.cuda.synchronize()
    assert torch.equal(again, ref)
    # two fp32 sums of the same products: one rounding to bf16 apart, and near zero what they lose to cancellation
    assert bool(((y.float() - ref.float()).abs() <= 2.0 ** -7 * ref.float().abs() + 1e-5).all())
    if polls == 0:
        assert not torch.equal(y, ref)                                             # (computed another way: some roundings differ)


def test_depthwise7_non_finite_pixels_reach_their_own_windows_only(either_kernel):
    N, H, W, C = 2, 20, 19, 64
    g = torch.Generator().manual_seed(synth.SEED_BASE + 7200)
    x = torch.randn((N, H, W, C), generator=g).to(torch.bfloat16)
    w = (torch.rand((7, 7, C), generator=g) * 0.1 + 0.05).to(torch.bfloat16)   # positive: an infinity keeps its sign
    bad = [(0, 5, 6, 3, float("inf")), (1, 10, 0, 7, float("nan")), (1, 19, 18, 40, float("-inf"))]
    clean = x.clone()
    for n, h, c0, c, v in bad:
        x[n, h, c0, c] = v
        clean[n, h, c0, c] = 0.0
    desc = api.make_desc(N, H, W, C, C, 7, 7, 1, 3, bias=False)
    y = api.ssconv_depthwise(desc, x.to(DEV), w.to(DEV)).cpu()
    y_clean = api.ssconv_depthwise(desc, clean.to(DEV), w.to(DEV)).cpu()
    touched = torch.zeros(y.shape, dtype=torch.bool)
    for n, h, c0, c, v in bad:
        box = (n, slice(max(0, h - 3), h + 4), slice(max(0, c0 - 3), c0 + 4), c)
        touched[box] = True
        assert bool(torch.isnan(y[box]).all()) if v != v else bool((y[box] == v).all())
    # outputs next to them are computed again on fp32 pipes in another order of summation: one bf16 rounding apart
    err = (y.float() - y_clean.float()).abs()[~touched]
    assert bool((err <= 2.0 ** -7 * y_clean.float().abs()[~touched] + 1e-5).all())


@pytest.mark.parametrize("data", ["normal", "spread", "positive"])
def test_depthwise7_sums_are_as_exact_as_fp32_ones(data):
    # The bias (added last) is minus the exact sum of one output per channel, so that what is left there is the error of
    # the sum.  (17 maps of 4 x 1 outputs: fewer, or flatter ones, would go to the fp32 kernel.)
    C, units = 4096, []
    for seed in range(8):
        g = torch.Generator().manual_seed(synth.SEED_BASE + 7900 + seed)
        x, w = torch.randn((17, 10, 7, C), generator=g), torch.randn((7, 7, C), generator=g) / 7
        if data == "spread":
            x = x * torch.exp(2.0 * torch.randn(x.shape, generator=g))
        if data == "positive":
            x, w = x.abs(), w.abs()
        x, w = x.to(torch.bfloat16), w.to(torch.bfloat16)
        n, row = 2 * seed, seed % 4
        products = x[n, row:row + 7].double() * w.double()
        total = products.sum((0, 1))
        bias = (-total).float()
        desc = api.make_desc(17, 10, 7, C, C, 7, 7, 1, 0, bias=True)
        y = api.ssconv_depthwise(desc, x.to(DEV), w.to(DEV), bias.to(DEV))[n, row, 0].cpu().double()
        units.append((y - (total + bias.double())) / products.abs().sum((0, 1)) * 2.0 ** 24)
    err = torch.cat(units)
    # what a chain of 49 fused multiply-adds leaves on these data (0.163, 0.744, 0.801 over 131072 sums; a fortieth more for
    # the sampling of a quarter as many)
    assert float(err.pow(2).mean().sqrt()) <= 1.025 * {"normal": 0.163, "spread": 0.744, "positive": 0.801}[data]
    assert abs(float(err.mean())) <= 0.3


@pytest.mark.parametrize("relu", [False, True], ids=["none", "relu"])
@pytest.mark.parametrize("with_bias", [False, True], ids=["no_bias", "bias"])
def test_depthwise7_non_finite_outputs_are_those_of_the_fp32_kernel(relu, with_bias, either_kernel):
    N, H, W, C = 3, 22, 25, 64
    g = torch.Generator(device=DEV).manual_seed(synth.SEED_BASE + 7250)
    x = torch.randn((N, H, W, C), generator=g, device=DEV).to(torch.bfloat16)
    w = (torch.randn((7, 7, C), generator=g, device=DEV) / 7).to(torch.bfloat16)
    bias = torch.randn(C, generator=g, device=DEV) if with_bias else None
    for n, h, c0, c, v in [(0, 5, 6, 3, float("inf")), (0, 6, 9, 3, float("-inf")), (1, 10, 0, 7, float("nan")), (2, 21, 24, 40, float("-inf")),
                           (1, 3, 3, 8, 3.0e38), (1, 3, 4, 8, 3.0e38)]:
        x[n, h, c0, c] = v
    desc = api.make_desc(N, H, W, C, C, 7, 7, 1, 3, bias=with_bias, relu=relu)
    y = api.ssconv_depthwise(desc, x, w, bias)
    api.ssconv_tune(api.TUNE_DEPTHWISE_MMA, 0)
    try:
        ref = api.ssconv_depthwise(desc, x, w, bias)
    finally:
        api.ssconv_tune(api.TUNE_DEPTHWISE_MMA, -1)
    assert torch.equal(torch.isnan(y), torch.isnan(ref)) and torch.equal(y == float("inf"), ref == float("inf"))
    assert torch.equal(y == float("-inf"), ref == float("-inf")) and not bool(torch.isfinite(ref).all())
    fin = torch.isfinite(ref)
    # (one bf16 rounding apart; the sums that meet 3e38 have lost everything below 2^-24 of it)
    near = fin.clone()
    near[1, :8, :9, 8] = False
    assert bool(((y.float() - ref.float()).abs()[near] <= 2.0 ** -7 * ref.float().abs()[near] + 1e-5).all())


@pytest.mark.parametrize("data", ["normal", "spread", "positive"])
def test_depthwise7_sums_on_small_maps_are_as_exact(data):
    # as above, on the kernel for small maps (1360 blocks); the bias is the first thing its sums hold
    C, units = 2560, []
    for seed in range(13):
        g = torch.Generator().manual_seed(synth.SEED_BASE + 7950 + seed)
        x, w = torch.randn((17, 10, 7, C), generator=g), torch.randn((7, 7, C), generator=g) / 7
        if data == "spread":
            x = x * torch.exp(2.0 * torch.randn(x.shape, generator=g))
        if data == "positive":
            x, w = x.abs(), w.abs()
        x, w = x.to(torch.bfloat16), w.to(torch.bfloat16)
        n, row = seed, seed % 4
        products = x[n, row:row + 7].double() * w.double()
        total = products.sum((0, 1))
        bias = (-total).float()
        desc = api.make_desc(17, 10, 7, C, C, 7, 7, 1, 0, bias=True)
        y = api.ssconv_depthwise(desc, x.to(DEV), w.to(DEV), bias.to(DEV))[n, row, 0].cpu().double()
        units.append((y - (total + bias.double())) / products.abs().sum((0, 1)) * 2.0 ** 24)
    err = torch.cat(units)
    print("small maps", data, float(err.pow(2).mean().sqrt()), float(err.mean()))
    # what the tensor-core kernel leaves on these data (a fortieth more for the sampling)
    assert float(err.pow(2).mean().sqrt()) <= 1.025 * {"normal": 0.156, "spread": 0.617, "positive": 0.730}[data]
    assert abs(float(err.mean())) <= 0.3
