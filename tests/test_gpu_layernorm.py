"""The layer norm for few pixels against the one for many (which the oracle checks): the same arithmetic, bit for bit."""
import pytest
import torch

from paper_2411_00288_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("C", [8, 24, 96, 192, 256, 384, 520, 768, 1024])
def test_few_pixels_as_many(C):
    g = torch.Generator(device=DEV).manual_seed(C)
    pixels = 300000 if C <= 192 else 30000            # more than three turns of every warp that the chip holds
    x = (torch.randn((pixels, C), generator=g, device=DEV) * 2 + 0.5).to(torch.bfloat16)
    gamma = 1.0 + 0.1 * torch.randn(C, generator=g, device=DEV)
    beta = 0.1 * torch.randn(C, generator=g, device=DEV)
    many = api.ssconv_layernorm(x, gamma, beta, 1e-6)
    for n in (1, 7, 33, 1000, 2961, 7001):
        buf = torch.full((n + 2, C), -5.0, dtype=torch.bfloat16, device=DEV)
        api.ssconv_layernorm(x[:n], gamma, beta, 1e-6, y=buf[1:n + 1])
        assert torch.equal(buf[1:n + 1], many[:n]), n
        assert bool((buf[0] == -5.0).all()) and bool((buf[-1] == -5.0).all())
