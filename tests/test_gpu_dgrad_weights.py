"""The input gradient reads the layer's own weights, as a transposed operand."""
import pytest
import torch

from paper_2411_00288_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# Ragged channels on either side, several channel tiles, resident weights
# (one channel tile, a shallow K), thread-block pairs, a K shared by the CTAs of a cluster, spread gradients
DGRAD = [
    ("ragged_both",     2, 9,  8,  72,  136, 3, 1, 1, 1),
    ("c_in_8",          2, 9,  9,  8,   64,  3, 1, 1, 1),
    ("c_out_8",         2, 9,  9,  64,  8,   3, 1, 1, 1),     # (the 8-channel mode: exchanged and reversed first)
    ("pointwise",       4, 28, 28, 96,  384, 1, 1, 0, 1),
    ("resident",        4, 28, 28, 64,  72,  1, 1, 0, 1),
    ("dilated_5x5",     1, 13, 11, 40,  48,  5, 1, 2, 2),
    ("pairs",           32, 28, 28, 256, 192, 3, 1, 1, 1),
    ("few_tiles",       1, 7,  7,  128, 512, 3, 1, 1, 1),
    ("spread",          2, 14, 14, 64,  72,  3, 2, 1, 2),
    ("unaligned_long",  16, 28, 28, 72, 512, 3, 1, 1, 1),     # (rows between sectors, a long K: rearranged first)
    ("unaligned_short", 5, 37, 37, 40,  512, 1, 1, 0, 1),
]


@pytest.mark.parametrize("case", DGRAD, ids=[c[0] for c in DGRAD])
def test_dgrad_reads_the_layers_own_weights(case):
    name, n, h, w, ci, co, k, s, p, dil = case
    g = torch.Generator().manual_seed(7000 + DGRAD.index(case))
    desc = api.make_desc(n, h, w, ci, co, k, k, stride=s, pad=p, dil=dil, bias=False)
    ho, wo = api.ssconv_out_shape(desc)
    wt = (torch.randn((co, k, k, ci), generator=g) / (k * k * co) ** 0.5).to(torch.bfloat16).to(DEV)
    dy = torch.randn((n, ho, wo, co), generator=g).to(torch.bfloat16).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    launches = api.ssconv_launch_count()
    dx = api.ssconv_dgrad(desc, dy, wt, dev_status=status)
    launches = api.ssconv_launch_count() - launches
    if name.startswith("unaligned"):
        assert launches == (2 if name == "unaligned_long" else 1)
    # every output pixel's gradient at the pixels that it was computed from, one matrix product per tap
    ref = torch.zeros((n, h + 2 * p, w + 2 * p, ci), dtype=torch.float64, device=DEV)
    for a in range(k):
        for b in range(k):
            ref[:, a * dil:a * dil + s * (ho - 1) + 1:s, b * dil:b * dil + s * (wo - 1) + 1:s] += dy.double() @ wt[:, a, b].double()
    ref = ref[:, p:p + h, p:p + w]
    assert int(status.item()) == 0
    err = (dx.double() - ref).abs()
    # one rounding to bf16 (2^-9 of the value) and fp32 sums of k * k * co products of variance 1 / (k * k * co)
    assert bool((err <= 2.0 ** -8 * ref.abs() + 1e-4).all()), float(err.max())
