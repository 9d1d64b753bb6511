"""Python binding of libssconv.so: the same entry points as include/ssconv.h.

Only argument marshalling happens here; torch supplies device memory and the current
stream.  The calls that a network makes per layer and step go through the native binding
(csrc/binding.cpp), which converts and checks their arguments; the others through ctypes.
There is no CPU path: if the library is missing or a call fails, an exception is raised.
"""
from __future__ import annotations

import ctypes
import functools
import importlib.util
import os
from dataclasses import dataclass
from typing import Optional, Tuple

import torch

FLAG_BIAS = 1
FLAG_RELU = 2
FLAG_GELU = 4
MASK_LOGITS_F32 = 0
MASK_MAGNITUDE_BF16 = 1
MASK_MAGNITUDE_E4M3 = 2
OK = 0
ERR_TIMEOUT = 8

_LIB_PATH = os.path.join(os.path.dirname(os.path.abspath(__file__)), "libssconv.so")
EXPORTS = ("ssconv_version", "ssconv_launch_count", "ssconv_status_string", "ssconv_out_shape", "ssconv_sizes",
           "ssconv_plan", "ssconv_plan_for_sms", "ssconv_tune", "ssconv_window_extent", "ssconv_selftest_wait_timeout", "ssconv_selftest_depthwise_give_up",
           "ssconv_select_mask", "ssconv_nm_patterns", "ssconv_select_mask_nm", "ssconv_apply_mask_nm",
           "ssconv_compress", "ssconv_decompress", "ssconv_maxpool", "ssconv_pad_channels", "ssconv_space_to_depth", "ssconv_unfold_w",
           "ssconv_fold_factor", "ssconv_fold_desc", "ssconv_fold_weights", "ssconv_forward", "ssconv_forward_res",
           "ssconv_forward_dense_res", "ssconv_forward_dense", "ssconv_forward_dense_strided",
           "ssconv_mask_norms", "ssconv_absmax", "ssconv_stability_threshold", "ssconv_soft_mask", "ssconv_mask_grad", "ssconv_adamw", "ssconv_dgrad_prepare", "ssconv_dgrad_spread", "ssconv_wgrad", "ssconv_wgrad_ws_bytes", "ssconv_dgrad", "ssconv_dgrad_ws_bytes",
           "ssconv_forward_static_ws",
           "ssconv_sizes_grouped", "ssconv_compress_grouped", "ssconv_forward_grouped", "ssconv_forward_dense_grouped",
           "ssconv_depthwise", "ssconv_layernorm",
           "ssconv_quantize_e4m3", "ssconv_sizes_fp8", "ssconv_compress_fp8", "ssconv_decompress_fp8",
           "ssconv_forward_fp8", "ssconv_forward_dense_fp8")


class SsconvError(RuntimeError):
    def __init__(self, fn: str, status: int, text: str):
        super().__init__(f"{fn} failed: status {status} ({text})")
        self.status = status


class Desc(ctypes.Structure):
    """Mirror of ssconv_desc_t."""
    _fields_ = [(n, ctypes.c_int32) for n in (
        "N", "H", "W", "C_in", "C_out", "KH", "KW", "stride_h", "stride_w", "pad_h", "pad_w", "dil_h", "dil_w")] + [
        ("flags", ctypes.c_uint32)]


def make_desc(N, H, W, C_in, C_out, KH, KW, stride=1, pad=0, dil=1, bias=True, relu=False, gelu=False) -> Desc:
    def pair(v):
        return (v, v) if isinstance(v, int) else tuple(v)
    (sh, sw), (ph, pw), (dh, dw) = pair(stride), pair(pad), pair(dil)
    flags = (FLAG_BIAS if bias else 0) | (FLAG_RELU if relu else 0) | (FLAG_GELU if gelu else 0)
    return Desc(N, H, W, C_in, C_out, KH, KW, sh, sw, ph, pw, dh, dw, flags)


def desc_from_spec(spec) -> Desc:
    """Descriptor for a synth.LayerSpec."""
    return make_desc(spec.N, spec.H, spec.W, spec.C_in, spec.C_out, spec.KH, spec.KW, spec.stride, spec.pad,
                     spec.dil, bias=spec.has_bias, relu=spec.relu and not spec.gelu, gelu=spec.gelu)


_lib = None


def _prototypes():
    """{entry point: (result, arguments)} as in include/ssconv.h.  Pointers (tensors, streams, descriptors and results
    alike) are passed as addresses."""
    vp, i32, i64, sz = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_size_t
    f32, f64 = ctypes.c_float, ctypes.c_double
    return {
        "ssconv_version": (i32, []),
        "ssconv_launch_count": (ctypes.c_uint64, []),
        "ssconv_status_string": (ctypes.c_char_p, [i32]),
        "ssconv_out_shape": (i32, [vp] * 3),
        "ssconv_sizes": (i32, [vp] * 6),
        "ssconv_plan": (i32, [vp, i32] + [vp] * 5),
        "ssconv_plan_for_sms": (i32, [vp, i32, i32] + [vp] * 5),
        "ssconv_tune": (i32, [i32, i32]),
        "ssconv_window_extent": (i32, [i32] * 5),
        "ssconv_selftest_wait_timeout": (i32, [i64, vp, vp]),
        "ssconv_select_mask": (i32, [i32, vp, i64, vp, vp]),
        "ssconv_nm_patterns": (i32, [i32, i32]),
        "ssconv_select_mask_nm": (i32, [i32, vp, i64, i32, i32, vp, vp]),
        "ssconv_apply_mask_nm": (i32, [vp, vp, i64, i32, i32, vp, vp]),
        "ssconv_compress": (i32, [vp] * 6),
        "ssconv_decompress": (i32, [vp] * 6),
        "ssconv_maxpool": (i32, [vp, vp] + [i32] * 7 + [vp]),
        "ssconv_pad_channels": (i32, [vp, vp, i64, i32, i32, vp]),
        "ssconv_space_to_depth": (i32, [vp, vp] + [i32] * 9 + [vp]),
        "ssconv_unfold_w": (i32, [vp, vp, i64] + [i32] * 7 + [vp]),
        "ssconv_fold_factor": (i32, [vp]),
        "ssconv_fold_desc": (i32, [vp, i32, vp]),
        "ssconv_fold_weights": (i32, [vp, i32, vp, vp, i64, vp, vp, vp]),
        "ssconv_forward": (i32, [vp] * 7 + [sz, vp, vp]),
        "ssconv_forward_res": (i32, [vp] * 8 + [sz, vp, vp]),
        "ssconv_forward_dense": (i32, [vp] * 6 + [sz, vp, vp]),
        "ssconv_forward_dense_res": (i32, [vp] * 7 + [sz, vp, vp]),
        "ssconv_forward_dense_strided": (i32, [vp, vp, i64, i64, i64, vp, vp, vp, vp, sz, vp, vp]),
        "ssconv_forward_static_ws": (i32, [vp] * 8),
        "ssconv_mask_norms": (i32, [vp, vp, i32, i64, vp, vp]),
        "ssconv_absmax": (i32, [vp, i64, vp, vp]),
        "ssconv_stability_threshold": (f64, [i32, f64, vp, i32, i32, f64, f64]),
        "ssconv_soft_mask": (i32, [vp, vp, f32, vp, i64, vp, vp, vp]),
        "ssconv_mask_grad": (i32, [vp, f32, vp, vp, i64, vp, vp]),
        "ssconv_adamw": (i32, [vp] * 4 + [i64, i32] + [f32] * 5 + [vp]),
        "ssconv_dgrad_prepare": (i32, [vp] * 5),
        "ssconv_dgrad_spread": (i32, [vp] * 4),
        "ssconv_wgrad": (i32, [vp] * 5 + [sz, vp, vp]),
        "ssconv_wgrad_ws_bytes": (i32, [vp, vp]),
        "ssconv_dgrad": (i32, [vp] * 5 + [sz, vp, vp]),
        "ssconv_dgrad_ws_bytes": (i32, [vp, vp]),
        "ssconv_sizes_grouped": (i32, [vp, i32, vp, vp, vp]),
        "ssconv_compress_grouped": (i32, [vp, i32] + [vp] * 5),
        "ssconv_forward_grouped": (i32, [vp, i32] + [vp] * 6 + [sz, vp, vp]),
        "ssconv_forward_dense_grouped": (i32, [vp, i32] + [vp] * 5 + [sz, vp, vp]),
        "ssconv_depthwise": (i32, [vp] * 6),
        "ssconv_selftest_depthwise_give_up": (i32, [vp] * 5 + [i32, vp]),
        "ssconv_layernorm": (i32, [vp, vp, vp, f32, vp, i64, i32, vp]),
        "ssconv_quantize_e4m3": (i32, [vp, vp, i64, f32, vp]),
        "ssconv_sizes_fp8": (i32, [vp] * 4),
        "ssconv_compress_fp8": (i32, [vp] * 6),
        "ssconv_decompress_fp8": (i32, [vp] * 6),
        "ssconv_forward_fp8": (i32, [vp] * 5 + [f32] + [vp] * 3),
        "ssconv_forward_dense_fp8": (i32, [vp] * 4 + [f32] + [vp] * 3),
    }


def lib():
    """Load libssconv.so once; raise if it has not been built."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise FileNotFoundError(
                f"{_LIB_PATH} is missing: build it with `python -m paper_2411_00288_b200.build` "
                "(there is no fallback path)")
        L = ctypes.CDLL(_LIB_PATH)
        for name, (restype, argtypes) in _prototypes().items():
            f = getattr(L, name)
            f.restype, f.argtypes = restype, argtypes
        _lib = L
    return _lib


_native = None


def _binding():
    """The native binding (csrc/binding.cpp), loaded once; raise if it has not been built for this torch and interpreter."""
    global _native
    if _native is None:
        lib()
        from .build import binding_path
        path = binding_path()
        if not os.path.exists(path):
            raise FileNotFoundError(
                f"{path} is missing: build it for torch {torch.__version__} with `python -m paper_2411_00288_b200.build` "
                "(there is no fallback path)")
        spec = importlib.util.spec_from_file_location(f"{__package__}._binding", path)
        native = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(native)
        _native = native
    return _native


def status_string(status: int) -> str:
    return lib().ssconv_status_string(status).decode()


def _check(fn: str, status: int):
    if status != OK:
        raise SsconvError(fn, status, status_string(status))


def _ptr(t: Optional[torch.Tensor]):
    return None if t is None else t.data_ptr()


def _raw_stream_functions(module):
    """(current raw stream of a device, current device) of a torch extension module, or None where this torch has not both:
    they are not public names."""
    names = ("_cuda_getCurrentRawStream", "_cuda_getDevice")
    found = tuple(getattr(module, n, None) for n in names)
    return None if None in found else found


_RAW = _raw_stream_functions(torch._C)


def _stream(stream=None):
    """The raw handle of a stream, or of the current device's current one (without a Stream object around it, which
    takes 3 us to make, where torch lets one)."""
    if stream is not None:
        return stream.cuda_stream
    if _RAW is None or not torch.cuda.is_initialized():
        return torch.cuda.current_stream().cuda_stream
    current, device = _RAW
    return current(device())


def _need_cuda(*tensors):
    for t in tensors:
        if t is not None and not (t.is_cuda and t.is_contiguous()):
            raise ValueError("tensors must be contiguous CUDA tensors")


def ssconv_version() -> int:
    return int(lib().ssconv_version())


def ssconv_launch_count() -> int:
    """Kernels launched by the library in this process so far."""
    return int(lib().ssconv_launch_count())


def ssconv_out_shape(desc: Desc) -> Tuple[int, int]:
    return _out_shape(bytes(desc))


# (by the descriptor's content: host arithmetic of the library, the same at every call)
@functools.lru_cache(maxsize=1024)
def _out_shape(desc_bytes: bytes) -> Tuple[int, int]:
    desc, h, w = Desc.from_buffer_copy(desc_bytes), ctypes.c_int32(), ctypes.c_int32()
    _check("ssconv_out_shape", lib().ssconv_out_shape(ctypes.byref(desc), ctypes.byref(h), ctypes.byref(w)))
    return int(h.value), int(w.value)


@dataclass(frozen=True)
class Sizes:
    G: int
    w_comp_bytes: int
    meta_bytes: int
    ws_bytes_sparse: int
    ws_bytes_dense: int


def ssconv_sizes(desc: Desc) -> Sizes:
    return _sizes(bytes(desc))


@functools.lru_cache(maxsize=1024)
def _sizes(desc_bytes: bytes) -> Sizes:
    desc, G = Desc.from_buffer_copy(desc_bytes), ctypes.c_int64()
    a, b, c, d = (ctypes.c_size_t() for _ in range(4))
    _check("ssconv_sizes", lib().ssconv_sizes(ctypes.byref(desc), ctypes.byref(G), ctypes.byref(a), ctypes.byref(b),
                                              ctypes.byref(c), ctypes.byref(d)))
    return Sizes(int(G.value), int(a.value), int(b.value), int(c.value), int(d.value))


def ssconv_select_mask(mode: int, scores: torch.Tensor, G: int, pattern: Optional[torch.Tensor] = None,
                       stream=None) -> torch.Tensor:
    """pattern uint8 [G] from fp32 scores [G,6] (mode LOGITS) or bf16 weights (mode MAGNITUDE)."""
    b = _binding()
    if pattern is None:
        _need_cuda(scores)
        pattern = b.blob(G, scores)
    _check("ssconv_select_mask", b.ssconv_select_mask(mode, scores, G, pattern, stream))
    return pattern


def ssconv_nm_patterns(N: int, M: int) -> int:
    """n = C(M, N), the number of N:M patterns (0 if N, M are out of the supported range)."""
    f = lib().ssconv_nm_patterns
    return int(f(int(N), int(M)))


def ssconv_select_mask_nm(mode: int, scores: torch.Tensor, G: int, N: int, M: int, stream=None) -> torch.Tensor:
    """pattern uint8 [G] for N:M blocks from fp32 scores [G, n] (mode LOGITS) or bf16 weights [G, M] (MAGNITUDE)."""
    _need_cuda(scores)
    pattern = torch.empty(G, dtype=torch.uint8, device=scores.device)
    f = lib().ssconv_select_mask_nm
    _check("ssconv_select_mask_nm", f(mode, _ptr(scores), G, N, M, _ptr(pattern), _stream(stream)))
    return pattern


def ssconv_apply_mask_nm(w: torch.Tensor, pattern: torch.Tensor, N: int, M: int, stream=None) -> torch.Tensor:
    """M .* W for an N:M mask: bf16 weights of w's shape with the dropped positions zeroed."""
    _need_cuda(w, pattern)
    out = torch.empty_like(w)
    f = lib().ssconv_apply_mask_nm
    _check("ssconv_apply_mask_nm", f(_ptr(w), _ptr(pattern), pattern.numel(), N, M, _ptr(out), _stream(stream)))
    return out


def ssconv_compress(desc: Desc, w: torch.Tensor, pattern: torch.Tensor, stream=None):
    """(w_comp, meta) uint8 blobs from bf16 weights [C_out,KH,KW,C_in] and pattern [G]."""
    b = _binding()
    _need_cuda(w)
    sz = ssconv_sizes(desc)
    w_comp, meta = b.blob(sz.w_comp_bytes, w), b.blob(sz.meta_bytes, w)
    _check("ssconv_compress", b.ssconv_compress(desc, w, pattern, w_comp, meta, stream))
    return w_comp, meta


def ssconv_decompress(desc: Desc, w_comp: torch.Tensor, meta: torch.Tensor, want_pattern: bool = True, stream=None):
    """(w_masked bf16 [C_out,KH,KW,C_in], pattern uint8 [G] or None) read back from the blobs."""
    _need_cuda(w_comp, meta)
    sz = ssconv_sizes(desc)
    w_out = torch.empty((desc.C_out, desc.KH, desc.KW, desc.C_in), dtype=torch.bfloat16, device=w_comp.device)
    pat = torch.empty(sz.G, dtype=torch.uint8, device=w_comp.device) if want_pattern else None
    _check("ssconv_decompress", lib().ssconv_decompress(ctypes.byref(desc), _ptr(w_comp), _ptr(meta), _ptr(w_out),
                                                        _ptr(pat), _stream(stream)))
    return w_out, pat


_workspaces = {}


def ssconv_window_extent(n: int, k: int, stride: int = 1, pad: int = 0, dil: int = 1) -> int:
    """Placements of a k-tap window along an axis of n elements, as the library computes them."""
    f = lib().ssconv_window_extent
    return int(f(int(n), int(k), int(stride), int(pad), int(dil)))


def ssconv_plan_for_sms(desc: Desc, sparse: bool, sm_count: int) -> dict:
    """ssconv_plan for a device with `sm_count` SMs; host arithmetic only, no GPU needed."""
    out = [ctypes.c_int32(0) for _ in range(5)]
    f = lib().ssconv_plan_for_sms
    _check("ssconv_plan_for_sms", f(ctypes.byref(desc), 1 if sparse else 0, int(sm_count), *[ctypes.byref(o) for o in out]))
    return dict(tile_positions=out[0].value, split=bool(out[1].value), ctas=out[2].value, ring_groups=out[3].value,
                pair=bool(out[4].value))


def ssconv_selftest_wait_timeout(limit_cycles: int, dev_status: torch.Tensor, stream=None) -> None:
    """Launch the one-block kernel whose bounded wait runs out; it stores ERR_TIMEOUT to dev_status."""
    _need_cuda(dev_status)
    f = lib().ssconv_selftest_wait_timeout
    _check("ssconv_selftest_wait_timeout", f(int(limit_cycles), _ptr(dev_status), _stream(stream)))


def ssconv_plan(desc: Desc, sparse: bool = True) -> dict:
    """Tile width, K split, thread blocks and ring depth the forward call would use on the current device."""
    out = [ctypes.c_int32(0) for _ in range(5)]
    f = lib().ssconv_plan
    _check("ssconv_plan", f(ctypes.byref(desc), 1 if sparse else 0, *[ctypes.byref(o) for o in out]))
    return dict(tile_positions=out[0].value, split=bool(out[1].value), ctas=out[2].value, ring_groups=out[3].value,
                pair=bool(out[4].value))


TUNE_TILE_POSITIONS, TUNE_PAIR, TUNE_WGRAD_RANGES, TUNE_WGRAD_PAIR, TUNE_RESIDENT_WEIGHTS, TUNE_PAIR_TILES = 1, 2, 3, 4, 5, 6
TUNE_DEPTHWISE_MMA = 7
TUNE_CLUSTER, TUNE_DEPTHWISE_SMALL = 8, 9


def ssconv_tune(option: int, value: int) -> None:
    """Process-wide planner override: TUNE_TILE_POSITIONS (0 = automatic, or a multiple of 16 in [48, 240]),
    TUNE_PAIR (-1 automatic, 0 never, 1 wherever thread-block pairs apply), TUNE_PAIR_TILES (-1 automatic, 0 one
    position tile per work item of the pair kernel, 1 two wherever they fit), the others as the header says."""
    f = lib().ssconv_tune
    _check("ssconv_tune", f(int(option), int(value)))


def default_workspace(device) -> torch.Tensor:
    """One scratch buffer per device, shared by calls that pass ws=None.  It needs no initialisation
    (the kernels write every part before reading it), so stream-ordered calls can share it; calls
    on different streams that may overlap must pass their own."""
    dev = device if isinstance(device, torch.device) else torch.device(device)
    key = dev.index if dev.index is not None else torch.cuda.current_device()
    if key not in _workspaces:
        nbytes = ssconv_sizes(make_desc(1, 8, 8, 8, 8, 1, 1)).ws_bytes_sparse
        _workspaces[key] = torch.empty(nbytes, dtype=torch.uint8, device=torch.device("cuda", key))
    return _workspaces[key]


def _alloc_y(desc: Desc, x: torch.Tensor) -> torch.Tensor:
    y = _binding().output(desc, x)
    if type(y) is int:
        _check("ssconv_out_shape", y)
    return y


def _scratch(x: torch.Tensor) -> torch.Tensor:
    """default_workspace of x's device."""
    ws = _workspaces.get(x.get_device())
    if ws is None:
        _need_cuda(x)
        ws = default_workspace(x.device)
    return ws


def ssconv_forward(desc: Desc, x: torch.Tensor, w_comp: torch.Tensor, meta: torch.Tensor,
                   bias: Optional[torch.Tensor] = None, y: Optional[torch.Tensor] = None,
                   ws: Optional[torch.Tensor] = None, dev_status: Optional[torch.Tensor] = None,
                   stream=None, residual: Optional[torch.Tensor] = None) -> torch.Tensor:
    """2:4 masked convolution forward; returns y bf16 [N,H_out,W_out,C_out] (enqueued, not synchronised).
    With `residual` (bf16, the shape of y) the call is ssconv_forward_res: y = act(bias + conv + residual)."""
    b = _binding()
    if ws is None:
        ws = _scratch(x)
    if y is None:
        y = _alloc_y(desc, x)
    if residual is None:
        _check("ssconv_forward", b.ssconv_forward(desc, x, w_comp, meta, bias, y, ws, ws, dev_status, stream))
    else:
        assert residual.shape == y.shape and residual.dtype == torch.bfloat16
        _check("ssconv_forward_res", b.ssconv_forward_res(desc, x, w_comp, meta, bias, residual, y, ws, ws, dev_status, stream))
    return y


def ssconv_forward_dense(desc: Desc, x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor] = None,
                         y: Optional[torch.Tensor] = None, ws: Optional[torch.Tensor] = None,
                         dev_status: Optional[torch.Tensor] = None, stream=None,
                         residual: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Dense counterpart with bf16 weights [C_out,KH,KW,C_in]; `residual` as in ssconv_forward."""
    b = _binding()
    if ws is None:
        ws = _scratch(x)
    if y is None:
        y = _alloc_y(desc, x)
    if residual is None:
        _check("ssconv_forward_dense", b.ssconv_forward_dense(desc, x, w, bias, y, ws, ws, dev_status, stream))
    else:
        assert residual.shape == y.shape and residual.dtype == torch.bfloat16
        _check("ssconv_forward_dense_res", b.ssconv_forward_dense_res(desc, x, w, bias, residual, y, ws, ws, dev_status, stream))
    return y


def ssconv_maxpool(x: torch.Tensor, k: int = 3, stride: int = 2, pad: int = 1, y: Optional[torch.Tensor] = None,
                   stream=None) -> torch.Tensor:
    """k x k max-pooling of NHWC bf16 activations; returns y [N,H_out,W_out,C] (enqueued, not synchronised)."""
    n, h, w, c = x.shape
    if y is None:
        _need_cuda(x)
        y = torch.empty((n, ssconv_window_extent(h, k, stride, pad), ssconv_window_extent(w, k, stride, pad), c),
                        dtype=torch.bfloat16, device=x.device)
    _check("ssconv_maxpool", _binding().ssconv_maxpool(x, y, n, h, w, c, k, stride, pad, stream))
    return y


def ssconv_space_to_depth(x: torch.Tensor, block: int, pad: int, Hb: int, Wb: int, C_pad: int,
                          y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """y [N,Hb,Wb,C_pad] with y[n,r,q,(bh*block+bw)*C+c] = x[n, block*r-pad+bh, block*q-pad+bw, c] (zeros outside
    the image and in the padding channels) from x [N,H,W,C] bf16."""
    n, h, w, c = x.shape
    if y is None:
        _need_cuda(x)
        y = torch.empty((n, Hb, Wb, C_pad), dtype=torch.bfloat16, device=x.device)
    _check("ssconv_space_to_depth", _binding().ssconv_space_to_depth(x, y, n, h, w, c, block, pad, Hb, Wb, C_pad, stream))
    return y


def ssconv_fold_factor(desc: Desc) -> int:
    """The number of neighbouring output pixels (1 or 2) the planner suggests folding into the output channels."""
    f = lib().ssconv_fold_factor
    return int(f(ctypes.byref(desc)))


def ssconv_fold_desc(desc: Desc, f: int) -> Desc:
    """Descriptor of the layer with f output pixels of a row folded into f * C_out output channels."""
    out = Desc()
    fn = lib().ssconv_fold_desc
    _check("ssconv_fold_desc", fn(ctypes.byref(desc), int(f), ctypes.byref(out)))
    return out


def ssconv_fold_weights(desc: Desc, f: int, w: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                        stream=None):
    """(w_folded, bias_folded) for ssconv_fold_desc(desc, f).  w: any tensor of C_out*KH*KW equal vectors (bf16 or
    e4m3 weights [C_out,KH,KW,C_in], patterns [G]); w_folded has the same dtype and f*C_out*KH*KW' vectors."""
    _need_cuda(w, bias)
    folded = ssconv_fold_desc(desc, f)
    w2 = b2 = None
    tap = 0
    if w is not None:
        vecs = desc.C_out * desc.KH * desc.KW
        assert w.is_contiguous() and w.numel() % vecs == 0
        per = w.numel() // vecs
        tap = per * w.element_size()
        w2 = torch.empty((folded.C_out, folded.KH, folded.KW, per), dtype=w.dtype, device=w.device)
        if w.dim() == 1:
            w2 = w2.view(-1)
    if bias is not None:
        assert bias.dtype == torch.float32
        b2 = torch.empty(folded.C_out, dtype=torch.float32, device=bias.device)
    fn = lib().ssconv_fold_weights
    _check("ssconv_fold_weights", fn(ctypes.byref(desc), int(f), _ptr(w), _ptr(w2), tap, _ptr(bias), _ptr(b2),
                                     _stream(stream)))
    return w2, b2


def ssconv_forward_dense_strided(desc: Desc, x: torch.Tensor, strides, w: torch.Tensor,
                                 bias: Optional[torch.Tensor] = None, y: Optional[torch.Tensor] = None,
                                 ws: Optional[torch.Tensor] = None, dev_status: Optional[torch.Tensor] = None,
                                 stream=None) -> torch.Tensor:
    """ssconv_forward_dense on a strided (possibly overlapping) view of x: `strides` = element strides of
    (w, h, n); pixel (n, h, w) of the input the descriptor names starts n*s_n + h*s_h + w*s_w elements into x."""
    b = _binding()
    if ws is None:
        ws = _scratch(x)
    if y is None:
        y = _alloc_y(desc, x)
    s_w, s_h, s_n = (int(v) for v in strides)
    _check("ssconv_forward_dense_strided",
           b.ssconv_forward_dense_strided(desc, x, s_w, s_h, s_n, w, bias, y, ws, ws, dev_status, stream))
    return y


def ssconv_pad_channels(x: torch.Tensor, C_pad: int, y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Zero-pad the channels of x [..., C] bf16 to C_pad (a multiple of 8); returns y [..., C_pad]."""
    _need_cuda(x, y)
    *lead, c = x.shape
    pixels = 1
    for d in lead:
        pixels *= d
    if y is None:
        y = torch.empty((*lead, C_pad), dtype=torch.bfloat16, device=x.device)
    f = lib().ssconv_pad_channels
    _check("ssconv_pad_channels", f(_ptr(x), _ptr(y), pixels, c, C_pad, _stream(stream)))
    return y


def ssconv_forward_static_ws(desc: Desc, x: torch.Tensor, w_comp: torch.Tensor, meta: torch.Tensor,
                             bias: Optional[torch.Tensor], y: torch.Tensor,
                             dev_status: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """ssconv_forward with the library's built-in scratch: for callers that must not allocate device
    memory.  Nothing is allocated here either, so the caller passes the output tensor y.  Small
    layers only (at most 64 output tiles); calls that overlap on the GPU race on the shared scratch."""
    _need_cuda(x, w_comp, meta, bias, y, dev_status)
    _check("ssconv_forward_static_ws", lib().ssconv_forward_static_ws(
        ctypes.byref(desc), _ptr(x), _ptr(w_comp), _ptr(meta), _ptr(bias), _ptr(y), _ptr(dev_status),
        _stream(stream)))
    return y


# ----------------------------------------------------------------------------- grouped / depthwise / layer norm
def ssconv_sizes_grouped(desc: Desc, groups: int):
    G = ctypes.c_int64()
    a, b = ctypes.c_size_t(), ctypes.c_size_t()
    f = lib().ssconv_sizes_grouped
    _check("ssconv_sizes_grouped", f(ctypes.byref(desc), groups, ctypes.byref(G), ctypes.byref(a), ctypes.byref(b)))
    return int(G.value), int(a.value), int(b.value)


def ssconv_compress_grouped(desc: Desc, groups: int, w: torch.Tensor, pattern: torch.Tensor, stream=None):
    """(w_comp, meta) of a grouped layer: the per-group blobs one after another."""
    _need_cuda(w, pattern)
    _, nv, nm = ssconv_sizes_grouped(desc, groups)
    w_comp = torch.empty(nv, dtype=torch.uint8, device=w.device)
    meta = torch.empty(nm, dtype=torch.uint8, device=w.device)
    f = lib().ssconv_compress_grouped
    _check("ssconv_compress_grouped", f(ctypes.byref(desc), groups, _ptr(w), _ptr(pattern), _ptr(w_comp), _ptr(meta),
                                        _stream(stream)))
    return w_comp, meta


def ssconv_forward_grouped(desc: Desc, groups: int, x: torch.Tensor, w_comp: torch.Tensor, meta: torch.Tensor,
                           bias: Optional[torch.Tensor] = None, y: Optional[torch.Tensor] = None,
                           dev_status: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """2:4 masked grouped convolution (one launch, or one per group on channel slices)."""
    b = _binding()
    ws = _scratch(x)
    if y is None:
        y = _alloc_y(desc, x)
    _check("ssconv_forward_grouped",
           b.ssconv_forward_grouped(desc, groups, x, w_comp, meta, bias, y, ws, ws, dev_status, stream))
    return y


def ssconv_forward_dense_grouped(desc: Desc, groups: int, x: torch.Tensor, w: torch.Tensor,
                                 bias: Optional[torch.Tensor] = None, y: Optional[torch.Tensor] = None,
                                 dev_status: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Dense grouped convolution; w bf16 [C_out, KH, KW, C_in/groups]."""
    b = _binding()
    ws = _scratch(x)
    if y is None:
        y = _alloc_y(desc, x)
    _check("ssconv_forward_dense_grouped", b.ssconv_forward_dense_grouped(desc, groups, x, w, bias, y, ws, ws, dev_status, stream))
    return y


def ssconv_depthwise(desc: Desc, x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor] = None,
                     y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Dense depthwise convolution; w bf16 tap-major [KH, KW, C]."""
    if y is None:
        _need_cuda(x)
        y = _alloc_y(desc, x)
    _check("ssconv_depthwise", _binding().ssconv_depthwise(desc, x, w, bias, y, stream))
    return y


def ssconv_selftest_depthwise_give_up(desc: Desc, x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor],
                                      polls: int, stream=None) -> torch.Tensor:
    """ssconv_depthwise with waits that run out after `polls` polls; the outputs are then computed again and come out whole."""
    _need_cuda(x, w, bias)
    y = _alloc_y(desc, x)
    _check("ssconv_selftest_depthwise_give_up", lib().ssconv_selftest_depthwise_give_up(
        ctypes.byref(desc), _ptr(x), _ptr(w), _ptr(bias), _ptr(y), int(polls), _stream(stream)))
    return y


def ssconv_layernorm(x: torch.Tensor, gamma: torch.Tensor, beta: torch.Tensor, eps: float = 1e-6,
                     y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Layer normalisation over the last axis of x (bf16), gamma / beta fp32 [C]."""
    c = x.shape[-1]
    if y is None:
        _need_cuda(x)
        y = torch.empty_like(x)
    _check("ssconv_layernorm", _binding().ssconv_layernorm(x, gamma, beta, eps, y, x.numel() // c, c, stream))
    return y


# ----------------------------------------------------------------------------- 8-bit (e4m3) operands
def ssconv_quantize_e4m3(x: torch.Tensor, scale: float = 1.0, y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """uint8 e4m3 codes of x * scale (x bf16, an even number of elements), nearest even, saturating."""
    _need_cuda(x)
    assert x.dtype == torch.bfloat16
    if y is None:
        y = torch.empty(x.shape, dtype=torch.uint8, device=x.device)
    _check("ssconv_quantize_e4m3", _binding().ssconv_quantize_e4m3(x, y, x.numel(), scale, stream))
    return y


def ssconv_sizes_fp8(desc: Desc):
    """(G, w_comp_bytes, meta_bytes) of the e4m3 blobs."""
    G = ctypes.c_int64()
    a, b = ctypes.c_size_t(), ctypes.c_size_t()
    f = lib().ssconv_sizes_fp8
    _check("ssconv_sizes_fp8", f(ctypes.byref(desc), ctypes.byref(G), ctypes.byref(a), ctypes.byref(b)))
    return int(G.value), int(a.value), int(b.value)


def ssconv_compress_fp8(desc: Desc, w: torch.Tensor, pattern: torch.Tensor, stream=None):
    """(w_comp, meta) uint8 blobs from e4m3 weights [C_out,KH,KW,C_in] (uint8) and pattern [G]."""
    _need_cuda(w, pattern)
    _, nv, nm = ssconv_sizes_fp8(desc)
    w_comp = torch.empty(nv, dtype=torch.uint8, device=w.device)
    meta = torch.empty(nm, dtype=torch.uint8, device=w.device)
    f = lib().ssconv_compress_fp8
    _check("ssconv_compress_fp8", f(ctypes.byref(desc), _ptr(w), _ptr(pattern), _ptr(w_comp), _ptr(meta), _stream(stream)))
    return w_comp, meta


def ssconv_decompress_fp8(desc: Desc, w_comp: torch.Tensor, meta: torch.Tensor, stream=None):
    """(w_masked uint8 e4m3 [C_out,KH,KW,C_in], pattern uint8 [G]) read back from the e4m3 blobs."""
    _need_cuda(w_comp, meta)
    G, _, _ = ssconv_sizes_fp8(desc)
    w_out = torch.empty((desc.C_out, desc.KH, desc.KW, desc.C_in), dtype=torch.uint8, device=w_comp.device)
    pat = torch.empty(G, dtype=torch.uint8, device=w_comp.device)
    f = lib().ssconv_decompress_fp8
    _check("ssconv_decompress_fp8", f(ctypes.byref(desc), _ptr(w_comp), _ptr(meta), _ptr(w_out), _ptr(pat), _stream(stream)))
    return w_out, pat


def ssconv_forward_fp8(desc: Desc, x: torch.Tensor, w_comp: torch.Tensor, meta: torch.Tensor,
                       bias: Optional[torch.Tensor] = None, out_scale: float = 1.0, y: Optional[torch.Tensor] = None,
                       dev_status: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """2:4 masked convolution on e4m3 activations (uint8 NHWC) and compressed e4m3 weights; bf16 output."""
    if y is None:
        _need_cuda(x)
        y = _alloc_y(desc, x)
    _check("ssconv_forward_fp8", _binding().ssconv_forward_fp8(desc, x, w_comp, meta, bias, out_scale, y, dev_status, stream))
    return y


def ssconv_forward_dense_fp8(desc: Desc, x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor] = None,
                             out_scale: float = 1.0, y: Optional[torch.Tensor] = None,
                             dev_status: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Dense counterpart on e4m3 weights [C_out,KH,KW,C_in] (uint8)."""
    if y is None:
        _need_cuda(x)
        y = _alloc_y(desc, x)
    _check("ssconv_forward_dense_fp8", _binding().ssconv_forward_dense_fp8(desc, x, w, bias, out_scale, y, dev_status, stream))
    return y


def ssconv_soft_mask(logits: torch.Tensor, noise: Optional[torch.Tensor], tau: float, w: Optional[torch.Tensor],
                     want_z: bool = True, want_w_eff: bool = True, stream=None,
                     z: Optional[torch.Tensor] = None, w_eff: Optional[torch.Tensor] = None):
    """(z fp32 [G,6] or None, w_eff bf16 shaped like w or None): relaxed choice (Eq. 3) and effective
    weights (Eq. 6 with the soft mask) of every group of four weights.  Output tensors may be passed in."""
    _need_cuda(logits, w)
    G = logits.shape[0]
    if z is None and want_z:
        z = torch.empty((G, 6), dtype=torch.float32, device=logits.device)
    if w_eff is None and want_w_eff:
        w_eff = torch.empty_like(w)
    _check("ssconv_soft_mask", _binding().ssconv_soft_mask(logits, noise, tau, w, G, z, w_eff, stream))
    return z, w_eff


def ssconv_mask_grad(z: torch.Tensor, tau: float, w: torch.Tensor, g_w_eff: torch.Tensor,
                     g_logits: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """dL/dlogits fp32 [G,6] from dL/dw_eff (fp32, the shape of w)."""
    _need_cuda(z)
    G = z.shape[0]
    if g_logits is None:
        g_logits = torch.empty((G, 6), dtype=torch.float32, device=z.device)
    _check("ssconv_mask_grad", _binding().ssconv_mask_grad(z, tau, w, g_w_eff, G, g_logits, stream))
    return g_logits


def ssconv_wgrad_ws_bytes(desc: Desc) -> int:
    n = ctypes.c_size_t()
    f = lib().ssconv_wgrad_ws_bytes
    _check("ssconv_wgrad_ws_bytes", f(ctypes.byref(desc), ctypes.byref(n)))
    return int(n.value)


def ssconv_wgrad(desc: Desc, x: torch.Tensor, dy: torch.Tensor, dw: Optional[torch.Tensor] = None,
                 ws: Optional[torch.Tensor] = None, dev_status: Optional[torch.Tensor] = None,
                 stream=None) -> torch.Tensor:
    """Weight gradient fp32 [C_out,KH,KW,C_in] of the layer from its bf16 input x and output gradient dy."""
    b = _binding()
    _need_cuda(x)
    if dw is None:
        dw = torch.empty((desc.C_out, desc.KH, desc.KW, desc.C_in), dtype=torch.float32, device=x.device)
    if ws is None:
        need = ssconv_wgrad_ws_bytes(desc)
        ws = b.blob(need, x) if need else None
    _check("ssconv_wgrad", b.ssconv_wgrad(desc, x, dy, dw, ws, ws, dev_status, stream))
    return dw


def ssconv_dgrad_ws_bytes(desc: Desc) -> int:
    n = ctypes.c_size_t()
    f = lib().ssconv_dgrad_ws_bytes
    _check("ssconv_dgrad_ws_bytes", f(ctypes.byref(desc), ctypes.byref(n)))
    return int(n.value)


def ssconv_dgrad(desc: Desc, dy: torch.Tensor, w: torch.Tensor, dx: Optional[torch.Tensor] = None,
                 ws: Optional[torch.Tensor] = None, dev_status: Optional[torch.Tensor] = None,
                 stream=None) -> torch.Tensor:
    """Input gradient bf16 [N,H,W,C_in] of the layer from its output gradient dy and bf16 weights, any stride."""
    b = _binding()
    _need_cuda(dy)
    if dx is None:
        dx = torch.empty((desc.N, desc.H, desc.W, desc.C_in), dtype=torch.bfloat16, device=dy.device)
    if ws is None:
        ws = b.blob(max(ssconv_dgrad_ws_bytes(desc), 16), dy)
    _check("ssconv_dgrad", b.ssconv_dgrad(desc, dy, w, dx, ws, ws, dev_status, stream))
    return dx


def ssconv_adamw(theta: torch.Tensor, g: torch.Tensor, m: torch.Tensor, v: torch.Tensor, step: int, lr: float = 1.0,
                 beta1: float = 0.9, beta2: float = 0.999, eps: float = 1e-8, weight_decay: float = 1e-4,
                 stream=None) -> torch.Tensor:
    """One AdamW update of fp32 parameters in place (theta, m, v are modified); step counts from 1."""
    _need_cuda(theta)
    assert theta.dtype == g.dtype == m.dtype == v.dtype == torch.float32
    assert theta.numel() == g.numel() == m.numel() == v.numel()
    _check("ssconv_adamw", _binding().ssconv_adamw(theta, g, m, v, theta.numel(), int(step), lr, beta1, beta2, eps,
                                                   weight_decay, stream))
    return theta


def ssconv_unfold_w(x: torch.Tensor, KW: int, stride: int = 1, pad: int = 0, dil: int = 1, C_pad: Optional[int] = None,
                    y: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Partial unfold along the width of x [..., W, C] bf16: y [..., W_out, C_pad] with
    y[..., wo, kw*C + c] = x[..., wo*stride - pad + kw*dil, c] (zeros outside and in padding channels)."""
    _need_cuda(x, y)
    *lead, w, c = x.shape
    rows = 1
    for d in lead:
        rows *= d
    if C_pad is None:
        C_pad = -(-KW * c // 64) * 64
    if y is None:
        y = torch.empty((*lead, ssconv_window_extent(w, KW, stride, pad, dil), C_pad), dtype=torch.bfloat16,
                        device=x.device)
    f = lib().ssconv_unfold_w
    _check("ssconv_unfold_w", f(_ptr(x), _ptr(y), rows, w, c, KW, stride, pad, dil, C_pad, _stream(stream)))
    return y


LEMMA_PERTURBATION, LEMMA_ANY_MASK, LEMMA_MASKED_UPDATE = 34, 35, 36


def ssconv_mask_norms(w: torch.Tensor, pattern: torch.Tensor, out: Optional[torch.Tensor] = None,
                      stream=None) -> torch.Tensor:
    """fp32 [3] on the device: ||W||_inf, ||(B-1).*W||_inf, ||B.*W||_inf (max absolute row sums; rows are
    output channels) for bf16 weights [C_out, ...] and one 2:4 pattern per group."""
    _need_cuda(w, pattern, out)
    c_out = w.shape[0]
    k = w.numel() // c_out
    if out is None:
        out = torch.empty((3,), dtype=torch.float32, device=w.device)
    f = lib().ssconv_mask_norms
    _check("ssconv_mask_norms", f(_ptr(w), _ptr(pattern), c_out, k, _ptr(out), _stream(stream)))
    return out


def ssconv_absmax(x: torch.Tensor, out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """fp32 [1] on the device: the largest magnitude in a bf16 tensor."""
    _need_cuda(x, out)
    if out is None:
        out = torch.empty((1,), dtype=torch.float32, device=x.device)
    f = lib().ssconv_absmax
    _check("ssconv_absmax", f(_ptr(x), x.numel(), _ptr(out), _stream(stream)))
    return out


def ssconv_stability_threshold(lemma: int, L: float, layer_norms, j: int, extra_norm: float, x_norm: float) -> float:
    """Confidence threshold of Lemma 3.4 / 3.5 / 3.6 (host arithmetic in the library)."""
    n = len(layer_norms)
    arr = (ctypes.c_double * n)(*[float(v) for v in layer_norms])
    f = lib().ssconv_stability_threshold
    v = float(f(lemma, float(L), arr, n, j, float(extra_norm), float(x_norm)))
    if v < 0:
        raise ValueError("bad arguments to ssconv_stability_threshold")
    return v


def ssconv_dgrad_prepare(desc: Desc, w: Optional[torch.Tensor], stream=None):
    """(desc_dx, w_t) for the input gradient of a layer: dx = ssconv_forward_dense(desc_dx, dy, w_t), with dy
    passed through ssconv_dgrad_spread first when the layer's stride is above 1.
    w_t bf16 [C_in,KH,KW,C_out] holds the reversed, channel-exchanged filter (None if w is None)."""
    _need_cuda(w)
    out = Desc()
    w_t = None
    if w is not None:
        w_t = torch.empty((desc.C_in, desc.KH, desc.KW, desc.C_out), dtype=torch.bfloat16, device=w.device)
    f = lib().ssconv_dgrad_prepare
    _check("ssconv_dgrad_prepare", f(ctypes.byref(desc), _ptr(w), _ptr(w_t), ctypes.byref(out), _stream(stream)))
    return out, w_t


def ssconv_dgrad_spread(desc: Desc, dy: torch.Tensor, stream=None) -> torch.Tensor:
    """dy [N,H_out,W_out,C_out] of a strided layer spread out with zeros to [N,Hz,Wz,C_out],
    Hz = H + 2 pad - dil (KH - 1): the input of the convolution ssconv_dgrad_prepare describes."""
    _need_cuda(dy)
    Hz = ssconv_window_extent(desc.H, desc.KH, 1, desc.pad_h, desc.dil_h)   # all unit-stride filter placements
    Wz = ssconv_window_extent(desc.W, desc.KW, 1, desc.pad_w, desc.dil_w)
    out = torch.empty((desc.N, Hz, Wz, desc.C_out), dtype=torch.bfloat16, device=dy.device)
    f = lib().ssconv_dgrad_spread
    _check("ssconv_dgrad_spread", f(ctypes.byref(desc), _ptr(dy), _ptr(out), _stream(stream)))
    return out
