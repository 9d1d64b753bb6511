"""The native binding's argument conversion, as far as it goes without a GPU."""
import ctypes

import pytest
import torch

from paper_2411_00288_b200 import api, build as libbuild


@pytest.fixture(scope="module")
def native():
    libbuild.build()
    return api._binding()


def test_entries_are_the_librarys_and_count_their_arguments(native):
    entries = [n for n in dir(native) if n.startswith("ssconv_")]
    assert len(entries) > 15 and set(entries) <= set(api.EXPORTS)
    for name in entries:
        expected = len(api._prototypes()[name][1])
        with pytest.raises(TypeError, match=f"{expected + 1} arguments, {expected} expected"):
            getattr(native, name)(*[None] * (expected + 1))


def test_tensors_that_the_library_cannot_take_are_refused(native):
    desc = api.make_desc(1, 8, 8, 64, 64, 3, 3, 1, 1)
    x = torch.zeros((1, 8, 8, 64), dtype=torch.bfloat16)
    for call in (lambda: api.ssconv_forward(desc, x, x, x, x), lambda: api.ssconv_select_mask(0, x, 4),
                 lambda: api.ssconv_depthwise(desc, x, x), lambda: api.ssconv_wgrad(desc, x, x),
                 lambda: api.ssconv_compress(desc, x, x), lambda: api.ssconv_layernorm(x, x, x),
                 lambda: api.ssconv_forward(desc, x, x, x, x, y=x, ws=x), lambda: api.ssconv_adamw(x.float(), x.float(), x.float(), x.float(), 1)):
        with pytest.raises(ValueError, match="contiguous CUDA tensors"):
            call()
    with pytest.raises(TypeError):
        native.ssconv_depthwise(desc, 16, 16, None, 16, None)      # addresses are not taken for tensors
    with pytest.raises(TypeError):
        native.ssconv_depthwise(b"\0" * 8, None, None, None, None, None)
    with pytest.raises(AttributeError):
        native.ssconv_depthwise(desc, None, None, None, None, 3)   # not a stream


def test_the_librarys_status_comes_back(native):
    ext = type("Stream", (), {"cuda_stream": 0})()
    desc = api.make_desc(1, 8, 8, 64, 64, 3, 3, 1, 1)
    assert native.ssconv_forward(desc, None, None, None, None, None, None, None, None, ext) == 1
    assert native.ssconv_select_mask(7, None, 4, None, ext) == 2
    assert native.output(api.make_desc(1, 8, 8, 64, 64, 3, 3, 0, 1), torch.zeros(1)) == 2
    y = native.output(api.make_desc(2, 8, 9, 64, 40, 3, 3, 2, 1), torch.zeros(1))
    assert y.shape == (2, 4, 5, 40) and y.dtype == torch.bfloat16
    assert native.blob(7, torch.zeros(1)).shape == (7,)
    assert ctypes.sizeof(api.Desc) == 56


def test_a_binding_built_for_another_torch_is_not_loaded(native, monkeypatch):
    monkeypatch.setattr(api, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(FileNotFoundError, match="python -m paper_2411_00288_b200.build"):
        api._binding()
    monkeypatch.undo()
    assert api._binding() is not None
