"""bf16 -> e4m3 at the ends of its 16-element vectors and on pointers that allow none, against torch's conversion."""
import pytest
import torch

from paper_2411_00288_b200 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [2, 14, 16, 18, 30, 32, 4098, 8192])
@pytest.mark.parametrize("x_off,y_off", [(0, 0), (2, 0), (0, 2), (8, 16), (10, 6)])
def test_quantize_vectors_tails_and_alignment(n, x_off, y_off):
    g = torch.Generator().manual_seed(synth.SEED_BASE + 7400 + n)
    xb = (torch.randn((n + x_off,), generator=g) * 60).to(torch.bfloat16).to(DEV)      # some beyond 448 after scaling
    x = xb[x_off:]
    yb = torch.full((n + y_off + 32,), 0xA5, dtype=torch.uint8, device=DEV)
    y = yb[y_off:y_off + n]
    api.ssconv_quantize_e4m3(x, 4.0, y=y)
    torch.cuda.synchronize()
    want = (x.float() * 4.0).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
    assert torch.equal(y, want)
    assert bool((yb[:y_off] == 0xA5).all()) and bool((yb[y_off + n:] == 0xA5).all())
