"""Kernels of one element or group per thread have two forms, by their number of blocks: what many blocks give is what slices
of few blocks give, bit for bit."""
import pytest
import torch

from paper_2411_00288_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
THREADS = 256


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV)


def _pieces(n, parts=5):
    """Slices of range(n) that start at multiples of a block."""
    step = (n // parts) // THREADS * THREADS
    return [slice(i * step, n if i == parts - 1 else (i + 1) * step) for i in range(parts)]


@pytest.mark.parametrize("blocks", [1184, 4096])
@pytest.mark.parametrize("extra", [0, 1], ids=["at_the_line", "one_more"])
def test_masks_of_many_groups_as_of_few(blocks, extra):
    g = torch.Generator(device=DEV).manual_seed(blocks)
    n = blocks * THREADS + extra
    logits, w, up = _randn(g, n, 6), _randn(g, n * 4).to(torch.bfloat16), _randn(g, n, 4)
    noise, codes = _randn(g, n, 6), torch.randint(0, 256, (n * 4,), generator=g, device=DEV, dtype=torch.uint8)
    z, w_eff = api.ssconv_soft_mask(logits, noise, 0.5, w)
    grad = api.ssconv_mask_grad(z, 0.5, w, up)
    choice = [api.ssconv_select_mask(m, t, n) for m, t in ((api.MASK_LOGITS_F32, logits), (api.MASK_MAGNITUDE_BF16, w),
                                                          (api.MASK_MAGNITUDE_E4M3, codes))]
    for s in _pieces(n):
        k, s4 = s.stop - s.start, slice(4 * s.start, 4 * s.stop)
        z_s, w_eff_s = api.ssconv_soft_mask(logits[s], noise[s], 0.5, w[s4])
        assert torch.equal(z_s, z[s]) and torch.equal(w_eff_s, w_eff[s4])
        assert torch.equal(api.ssconv_mask_grad(z_s, 0.5, w[s4], up[s]), grad[s])
        for m, t, c in ((api.MASK_LOGITS_F32, logits[s], choice[0]), (api.MASK_MAGNITUDE_BF16, w[s4], choice[1]),
                        (api.MASK_MAGNITUDE_E4M3, codes[s4], choice[2])):
            assert torch.equal(api.ssconv_select_mask(m, t, k), c[s])


@pytest.mark.parametrize("n", [4096 * THREADS * 16 + 2, 4096 * THREADS * 4 + 3], ids=["quantise", "adamw"])
def test_elementwise_calls_of_many_elements_as_of_few(n):
    g = torch.Generator(device=DEV).manual_seed(n)
    if n % 2 == 0:
        x = (_randn(g, n) * 200).to(torch.bfloat16)
        y = api.ssconv_quantize_e4m3(x, 1.5)
        assert all(torch.equal(api.ssconv_quantize_e4m3(x[s], 1.5), y[s]) for s in _pieces(n))
        return
    t, grad, m, v = _randn(g, n), _randn(g, n), _randn(g, n) * 0.1, _randn(g, n).abs() * 0.01
    parts = [tuple(p[s].clone() for p in (t, grad, m, v)) for s in _pieces(n)]
    api.ssconv_adamw(t, grad, m, v, 3, lr=1e-2)
    for s, (t_s, grad_s, m_s, v_s) in zip(_pieces(n), parts):
        api.ssconv_adamw(t_s, grad_s, m_s, v_s, 3, lr=1e-2)
        assert torch.equal(t_s, t[s]) and torch.equal(m_s, m[s]) and torch.equal(v_s, v[s])


def test_packing_of_many_weights_as_of_few():
    g = torch.Generator(device=DEV).manual_seed(5)
    ci, co = 33016, 1024                                         # 4128 blocks in all, 516 for 128 channels
    w = _randn(g, co, 1, 1, ci).to(torch.bfloat16)
    pattern = torch.randint(0, 6, (w.numel() // 4,), generator=g, device=DEV, dtype=torch.uint8)
    w_comp, meta = api.ssconv_compress(api.make_desc(1, 8, 8, ci, co, 1, 1), w, pattern)
    one = api.make_desc(1, 8, 8, ci, 128, 1, 1)
    parts = [api.ssconv_compress(one, w[c:c + 128], pattern[c * ci // 4:(c + 128) * ci // 4]) for c in range(0, co, 128)]
    assert torch.equal(w_comp, torch.cat([p[0] for p in parts])) and torch.equal(meta, torch.cat([p[1] for p in parts]))


def test_input_gradient_interleaved_by_many_blocks():
    n, h, ci, co = 11, 57, 256, 64                               # 4468 blocks of the gather kernel
    g = torch.Generator(device=DEV).manual_seed(6)
    desc = api.make_desc(n, h, h, ci, co, 3, 3, stride=2, pad=1, bias=False)
    ho = (h - 1) // 2 + 1
    w = (_randn(g, co, 3, 3, ci) / 24).to(torch.bfloat16)        # 24^2 = 9 co
    dy = _randn(g, n, ho, ho, co).to(torch.bfloat16)
    dx = api.ssconv_dgrad(desc, dy, w)
    ref = torch.zeros((n, h + 2, h + 2, ci), dtype=torch.float64, device=DEV)
    for a in range(3):
        for b in range(3):
            ref[:, a:a + 2 * ho - 1:2, b:b + 2 * ho - 1:2] += dy.double() @ w[:, a, b].double()
    ref = ref[:, 1:-1, 1:-1]
    # one rounding to bf16 (2^-9 of the value) and fp32 sums of at most 4 co products of variance 1 / (9 co)
    assert bool(((dx.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all())
