"""The layer norm for few pixels against the one for many (which the oracle checks): the same arithmetic, bit for bit."""
import pytest
import torch

from paper_2411_00288_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lanes(C):
    """Lanes that share a pixel: the library's choice."""
    c8 = C // 8
    g = next(g for g in (32, 16, 8, 4, 2, 1) if c8 % g == 0)
    return g if c8 // g <= 4 else next(g for g in (1, 2, 4, 8, 16, 32) if g >= c8 or g == 32)


@pytest.mark.parametrize("C", [8, 24, 32, 64, 96, 192, 256, 384, 520, 768, 1024])
def test_few_pixels_as_many(C):
    g = torch.Generator(device=DEV).manual_seed(C)
    per_warp, sms = 32 // _lanes(C), torch.cuda.get_device_properties(0).multi_processor_count
    # an SM holds three to nine blocks of four warps, by the form; never more than its 64 warps
    least, pixels = 4 * 3 * sms * per_warp, 4 * 64 * sms * per_warp   # (the latter: more than three turns of any form)
    x = (torch.randn((pixels, C), generator=g, device=DEV) * 2 + 0.5).to(torch.bfloat16)
    gamma = 1.0 + 0.1 * torch.randn(C, generator=g, device=DEV)
    beta = 0.1 * torch.randn(C, generator=g, device=DEV)
    many = api.ssconv_layernorm(x, gamma, beta, 1e-6)
    # a few pixels, then ragged numbers of them: one, two and three turns of every form
    for n in (1, 7, 33, 1000, 2961, 7001, *(k * least // 2 - per_warp - 1 for k in range(3, 19, 2))):
        buf = torch.full((n + 2, C), -5.0, dtype=torch.bfloat16, device=DEV)
        api.ssconv_layernorm(x[:n], gamma, beta, 1e-6, y=buf[1:n + 1])
        assert torch.equal(buf[1:n + 1], many[:n]), n
        assert bool((buf[0] == -5.0).all()) and bool((buf[-1] == -5.0).all())
