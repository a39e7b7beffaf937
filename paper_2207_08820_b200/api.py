"""Thin Python binding over the C ABI of ``include/bitserial.h``.

Argument marshalling only: tensors are torch CUDA tensors used as device buffers, streams are torch
streams, and every function forwards to the entry point of the same name.  No arithmetic of the method
happens here and nothing falls back to PyTorch ops.
"""
from __future__ import annotations

import ctypes
from typing import Optional

import torch

from ._lib import BitserialError, ConvParams, lib, native

UNSIGNED, SIGNED, BIPOLAR = 0, 1, 2
SIGNED_NIBBLES = 3      # signed filters of three bits prepared as nibbles; only where prepared filters are
NCHW, NHWC = 0, 1
ERR_UNSUPPORTED = 2

launch_count = 0   # kernels enqueued through this binding (one by every entry point below but chains and sequences of layers)


def _stream_ptr(stream: Optional[torch.cuda.Stream]) -> int:
    s = stream if stream is not None else torch.cuda.current_stream()
    return s.cuda_stream


def _ptr(t: Optional[torch.Tensor]) -> Optional[int]:
    if t is None:
        return None
    if not t.is_cuda or not t.is_contiguous():
        raise ValueError("expected a contiguous CUDA tensor")
    return t.data_ptr()


def _check(status: int, where: str) -> None:
    global launch_count
    if status != 0:
        raise BitserialError(status, where)
    launch_count += 1


def packed_act_words(N, C, H, W, bits) -> int:
    return lib().bs_packed_act_bytes(N, C, H, W, bits) // 4


def packed_wgt_words(O, C, R, S, bits) -> int:
    return lib().bs_packed_wgt_bytes(O, C, R, S, bits) // 4


def packed_rows_words(rows, K, bits) -> int:
    return lib().bs_packed_rows_bytes(rows, K, bits) // 4


def _words(n: int, device) -> torch.Tensor:
    return torch.empty(n, dtype=torch.int32, device=device)


def bitpack_activations(x: torch.Tensor, act_scale: float, a_bits: int, a_sign: int = UNSIGNED,
                        layout: int = NCHW, out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """x: float32 or int8 (codes), [N,C,H,W] (NCHW) or [N,H,W,C] (NHWC).  Returns int32 words
    viewed as [N, H, W, Cw, a_bits]."""
    st, out, _ = native().bitpack(x, act_scale, a_bits, a_sign, layout, out, stream)
    _check(st, "bitpack_activations")
    return out


def bitpack_operands(x: torch.Tensor, act_scale: float, a_bits: int, out: torch.Tensor, operands: int, stream=None) -> None:
    """:func:`bitpack_activations` of a float32 NCHW tensor to unsigned codes that writes, beside ``out``, the operand tensor ``operands`` of a bound
    sequence (``bs_sequence_input``)."""
    _check(native().bitpack_operands(x, act_scale, a_bits, out, operands, stream)[0], "bitpack_activations_operands")


def bitunpack_activations(packed: torch.Tensor, C: int, a_bits: int, a_sign: int = UNSIGNED, layout: int = NCHW,
                          stream=None) -> torch.Tensor:
    N, H, W, Cw, b = packed.shape
    shape = (N, C, H, W) if layout == NCHW else (N, H, W, C)
    out = torch.empty(shape, dtype=torch.int8, device=packed.device)
    st = lib().bitunpack_activations(_ptr(packed), N, C, H, W, a_bits, a_sign, layout, _ptr(out), _stream_ptr(stream))
    _check(st, "bitunpack_activations")
    return out


def pack_weights(w_codes: torch.Tensor, w_bits: int, w_sign: int, layout: int = NCHW, stream=None) -> torch.Tensor:
    """w_codes int8 [O,C,R,S] (layout NCHW = OIHW) or [O,R,S,C].  Returns int32 words [O,R,S,Cw,w_bits]."""
    if layout == NCHW:
        O, C, R, S = w_codes.shape
    else:
        O, R, S, C = w_codes.shape
    Cw = (C + 31) // 32
    out = _words(O * R * S * Cw * w_bits, w_codes.device)
    st = lib().pack_weights(_ptr(w_codes), layout, O, C, R, S, w_bits, w_sign, _ptr(out), _stream_ptr(stream))
    _check(st, "pack_weights")
    return out.view(O, R, S, Cw, w_bits)


def bs_pack_rows(codes: torch.Tensor, bits: int, sign: int, stream=None) -> torch.Tensor:
    rows, K = codes.shape
    Kw = (K + 31) // 32
    out = _words(rows * Kw * bits, codes.device)
    st = lib().bs_pack_rows(_ptr(codes), rows, K, bits, sign, _ptr(out), _stream_ptr(stream))
    _check(st, "bs_pack_rows")
    return out.view(rows, Kw, bits)


def bitserial_conv2d(act_packed: torch.Tensor, wgt_packed: torch.Tensor, *, C: int, stride: int = 1, pad: int = 0,
                     a_sign: int = UNSIGNED, w_sign: int = SIGNED, scale: Optional[torch.Tensor] = None,
                     bias: Optional[torch.Tensor] = None, relu: bool = False, out_bits: int = 0,
                     out_sign: int = UNSIGNED, residual: Optional[torch.Tensor] = None, res_scale: float = 0.0,
                     res_bits: int = 0, res_sign: int = UNSIGNED, res_c_offset: int = 0, res_c_total: int = 0,
                     out_i32: Optional[torch.Tensor] = None, want_i32: bool = False, i32_layout: int = NCHW,
                     out_packed: Optional[torch.Tensor] = None, out_c_offset: int = 0, out_c_total: int = 0,
                     workspace: Optional[torch.Tensor] = None, wgt_tc: Optional[torch.Tensor] = None, chained: bool = False,
                     stream=None):
    """act_packed [N,H,W,Cw,a_bits], wgt_packed [O,R,S,Cw,w_bits].  Returns (out_i32 or None, out_packed or None).
    A packed output is produced when ``out_bits`` > 0 (allocated here unless ``out_packed`` is given).
    ``workspace`` (zeroed device tensor, see :func:`conv_workspace`) lets the popcount kernels split the reduction
    (``bitserial_conv2d_ws``; the tensor-core kernel leaves it alone).
    ``wgt_tc`` (from :func:`tc_prepare_weights`) selects the tensor-core entry point ``bitserial_conv2d_tc``;
    with ``chained`` it is ``bitserial_conv2d_tc_chained`` (set-up overlaps the preceding kernel of the stream: filters,
    scale and bias must have been final before that kernel was launched)."""
    st, out_i32, out_packed = native().conv2d(
        act_packed, wgt_packed, C, stride, pad, a_sign, w_sign, scale, bias, relu, out_bits, out_sign, residual, res_scale, res_bits,
        res_sign, res_c_offset, res_c_total, out_i32, want_i32, i32_layout, out_packed, out_c_offset, out_c_total, workspace, wgt_tc,
        chained, stream)
    _check(st, "bitserial_conv2d")
    return out_i32, out_packed


def bitserial_gemm(a_packed: torch.Tensor, w_packed: torch.Tensor, K: int, *, a_sign: int = UNSIGNED,
                   w_sign: int = SIGNED, scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None,
                   relu: bool = False, out_bits: int = 0, out_sign: int = UNSIGNED,
                   out_i32: Optional[torch.Tensor] = None, want_i32: bool = True,
                   out_packed: Optional[torch.Tensor] = None, workspace: Optional[torch.Tensor] = None, stream=None):
    """a_packed [M,Kw,a_bits], w_packed [N,Kw,w_bits].  Returns (out_i32 [M,N] or None, out_packed or None).
    ``workspace`` (zeroed device tensor, see :func:`gemm_workspace`) lets the popcount kernels split the reduction
    (``bitserial_gemm_ws``; the tensor-core kernel leaves it alone)."""
    st, out_i32, out_packed = native().gemm(a_packed, w_packed, -1, -1, K, a_sign, w_sign, scale, bias, relu, out_bits, out_sign,
                                            out_i32, want_i32, out_packed, workspace, stream)
    _check(st, "bitserial_gemm")
    return out_i32, out_packed


def tc_prepare_weights(wgt_packed: torch.Tensor, C: int, w_sign: int, a_bits: int, stream=None) -> torch.Tensor:
    """Packed weights [O,R,S,Cw,w_bits] -> filter tiles for the tensor-core entry points, made for layers of ``a_bits`` activation bits (nibbles where
    both widths are at most 2, int8 otherwise; layers that need the other form take these too and convert them in each launch, more slowly).
    Signed filters of three bits for one or two bits are both, int8 and then nibbles, in a tensor of twice the size: layers of every width read
    their form as it is."""
    O, R, S, Cw, w_bits = wgt_packed.shape
    nbytes = lib().bs_tc_weights_bytes(O, C, R, S)
    if nbytes == 0:
        raise BitserialError(2, "bs_tc_weights_bytes")
    signs = [w_sign, SIGNED_NIBBLES] if w_bits == 3 and w_sign == SIGNED and a_bits <= 2 and C * R * S * 28 < 4000000 else [w_sign]
    out = torch.empty(nbytes * len(signs), dtype=torch.int8, device=wgt_packed.device)
    for k, sign in enumerate(signs):
        st = lib().bs_tc_prepare_weights(_ptr(wgt_packed), O, C, R, S, w_bits, sign, a_bits, _ptr(out) + k * nbytes, _stream_ptr(stream))
        _check(st, "bs_tc_prepare_weights")
    return out


def tc_weights_form(w_tc: Optional[torch.Tensor], wgt_shape, C: int, w_sign: int, a_bits: int):
    """(part of ``w_tc`` that layers of ``a_bits`` activation bits read, ``bs_sign_t`` that goes with it)."""
    O, R, S, _, w_bits = wgt_shape
    if w_tc is not None and w_bits == 3 and w_sign == SIGNED and a_bits <= 2:
        n = lib().bs_tc_weights_bytes(O, C, R, S)
        if w_tc.numel() * w_tc.element_size() == 2 * n:
            return w_tc.view(-1)[w_tc.numel() // 2:], SIGNED_NIBBLES
    return w_tc, w_sign


def tc_weights_read(w_tc: torch.Tensor, wgt_shape, C: int, a_bits: int):
    """What layers of ``a_bits`` activation bits read of filters prepared for them: a list of views."""
    O, R, S, _, w_bits = wgt_shape
    w_tc, sign = tc_weights_form(w_tc, wgt_shape, C, SIGNED, a_bits)
    n = lib().bs_tc_weights_read_bytes(O, C, R, S, 2 if sign == SIGNED_NIBBLES else w_bits, a_bits)     # (nibbles are laid out as those of two bits)
    if w_bits == 3 and n:
        w_tc = w_tc[:lib().bs_tc_weights_bytes(O, C, R, S)]
    return [w_tc] if n in (0, w_tc.numel()) else [w_tc[:n], w_tc[-16:]]


def tc_supported(N, C, H, W, O, k, stride, pad, a_bits, a_sign, w_bits, w_sign) -> bool:
    p = ConvParams(N=N, C=C, H=H, W=W, O=O, R=k, S=k, stride=stride, pad=pad, a_bits=a_bits, a_sign=a_sign,
                   w_bits=w_bits, w_sign=w_sign)
    return bool(lib().bs_tc_supported(ctypes.byref(p)))


def conv_params(act_shape, wgt_shape, *, C: int, stride: int = 1, pad: int = 0, a_sign: int = UNSIGNED, w_sign: int = SIGNED,
                scale: Optional[torch.Tensor] = None, bias: Optional[torch.Tensor] = None, relu: bool = False, out_bits: int = 0,
                out_sign: int = UNSIGNED, residual: Optional[torch.Tensor] = None, res_scale: float = 0.0, res_bits: int = 0,
                res_sign: int = UNSIGNED) -> ConvParams:
    """``bs_conv_params`` of a layer whose packed output is a whole tensor (no channel offset), from the shapes of the packed
    operands; for :func:`tc_chain_workspace_bytes` and :func:`bitserial_conv2d_tc_chain`."""
    N, H, W, Cw, a_bits = act_shape
    O, R, S, Cw2, w_bits = wgt_shape
    if Cw != Cw2 or Cw != (C + 31) // 32:
        raise ValueError("channel words of activations and weights disagree")
    return ConvParams(N=N, C=C, H=H, W=W, O=O, R=R, S=S, stride=stride, pad=pad, a_bits=a_bits, a_sign=a_sign, w_bits=w_bits,
                      w_sign=w_sign, scale=_ptr(scale), bias=_ptr(bias), relu=int(relu), out_bits=out_bits, out_sign=out_sign,
                      residual=_ptr(residual), res_scale=res_scale, res_bits=res_bits, res_sign=res_sign, res_c_offset=0,
                      res_c_total=O, out_c_offset=0, out_c_total=O, i32_layout=NCHW)


def _params_array(params):
    arr = (ConvParams * len(params))()
    for k, q in enumerate(params):
        ctypes.memmove(ctypes.addressof(arr[k]), ctypes.addressof(q), ctypes.sizeof(ConvParams))
    return arr


def tc_chain_workspace_bytes(params) -> int:
    """Bytes of the workspace ``bitserial_conv2d_tc_chain`` asks for with these layers; 0 when they cannot run as one chain."""
    return int(lib().bs_tc_chain_workspace_bytes(_params_array(params), len(params)))


def bitserial_conv2d_tc_chain(acts, wgts_tc, params, outs, workspace: torch.Tensor, chained: bool = False, stream=None) -> None:
    """Several same-shaped layers in one call, a launch each (``bitserial_conv2d_tc_chain``): per layer the packed input, the prepared
    filters, the :func:`conv_params` and the packed output tensor.  ``workspace``: device tensor of
    :func:`tc_chain_workspace_bytes` bytes."""
    global launch_count
    n = len(params)
    vp = ctypes.c_void_p * n
    st = lib().bitserial_conv2d_tc_chain(n, vp(*[_ptr(t) for t in acts]), vp(*[_ptr(t) for t in wgts_tc]), _params_array(params),
                                         vp(*[_ptr(t) for t in outs]), _ptr(workspace), workspace.numel() * workspace.element_size(),
                                         int(chained), _stream_ptr(stream))
    _check(st, "bitserial_conv2d_tc_chain")
    launch_count += n - 1


def run_sequence(sequence, launches: int, stream=None, ready: Optional[int] = None) -> None:
    """One pass of a bound sequence of layers (``bs_sequence_run``), which enqueues ``launches`` kernels.  ``ready``: its operand tensor that is up
    to date (``bs_sequence_run_ready``)."""
    global launch_count
    _check(native().sequence_run(sequence, stream, ready), "bs_sequence_run")
    launch_count += launches - 1


def bitserial_gemm_tc(a_packed: torch.Tensor, w_tc: torch.Tensor, N: int, K: int, w_bits: int, *, a_sign: int = UNSIGNED,
                      w_sign: int = SIGNED, scale=None, bias=None, relu: bool = False, out_bits: int = 0,
                      out_sign: int = UNSIGNED, want_i32: bool = True, out_i32: Optional[torch.Tensor] = None,
                      out_packed: Optional[torch.Tensor] = None, stream=None):
    """Tensor-core matrix product: a_packed [M,Kw,a_bits], w_tc from tc_prepare_weights on the [N,1,1,Kw,w_bits] rows."""
    st, out_i32, out_packed = native().gemm(a_packed, w_tc, N, w_bits, K, a_sign, w_sign, scale, bias, relu, out_bits, out_sign,
                                            out_i32, want_i32, out_packed, None, stream)
    _check(st, "bitserial_gemm_tc")
    return out_i32, out_packed


def gemm_workspace(M: int, N: int, K: int, a_bits: int, a_sign: int, w_bits: int, w_sign: int, device="cuda"):
    """Zeroed workspace for the reduction split of this matrix product, or None when the popcount planner would not split."""
    nbytes = lib().bs_gemm_workspace_bytes(M, N, K, a_bits, a_sign, w_bits, w_sign)
    return torch.zeros((nbytes + 3) // 4, dtype=torch.int32, device=device) if nbytes else None


def conv_workspace(N: int, C: int, H: int, W: int, O: int, k: int, stride: int, pad: int, a_bits: int, a_sign: int,
                   w_bits: int, w_sign: int, device="cuda"):
    """Zeroed workspace for the reduction split of this convolution, or None when the popcount planner would not split."""
    p = ConvParams(N=N, C=C, H=H, W=W, O=O, R=k, S=k, stride=stride, pad=pad, a_bits=a_bits, a_sign=a_sign,
                   w_bits=w_bits, w_sign=w_sign)
    nbytes = lib().bs_conv_workspace_bytes(ctypes.byref(p))
    return torch.zeros((nbytes + 3) // 4, dtype=torch.int32, device=device) if nbytes else None


def conv2d_f32(x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor] = None, stride: int = 1, pad: int = 0, relu: bool = False,
               out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Floating-point convolution of the layers kept in FP32 (``bs_conv2d_f32``): x [N,C,H,W], w [O,C,R,S] float32."""
    N, C, H, W = x.shape
    O, C2, R, S = w.shape
    if C != C2 or x.dtype != torch.float32 or w.dtype != torch.float32:
        raise ValueError("float32 tensors with matching channels expected")
    P, Q = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    if out is None:
        out = torch.empty(N, O, P, Q, dtype=torch.float32, device=x.device)
    _check(lib().bs_conv2d_f32(_ptr(x), _ptr(w), _ptr(bias), N, C, H, W, O, R, S, stride, pad, int(relu), _ptr(out), _stream_ptr(stream)),
           "bs_conv2d_f32")
    return out


def maxpool2d_f32(x: torch.Tensor, k: int, stride: int, pad: int, out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    N, C, H, W = x.shape
    P, Q = (H + 2 * pad - k) // stride + 1, (W + 2 * pad - k) // stride + 1
    if out is None:
        out = torch.empty(N, C, P, Q, dtype=torch.float32, device=x.device)
    _check(lib().bs_maxpool2d_f32(_ptr(x), N, C, H, W, k, stride, pad, _ptr(out), _stream_ptr(stream)), "bs_maxpool2d_f32")
    return out


def stem_codes_f32(x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor], act_scale: float, a_bits: int, out: torch.Tensor,
                   stream=None, operands: Optional[int] = None) -> bool:
    """Stem convolution (stride 2, pad 3) with ReLU, 3x3 stride-2 max pooling and quantise + pack in one call (``bs_stem_codes_f32``): images to the
    packed codes of :func:`conv2d_f32`, :func:`maxpool2d_f32` and :func:`bitpack_activations`.  False where the library has no such kernel for
    the shape: nothing was launched.  ``operands``: the operand tensor of ``out`` (``bs_sequence_input``), written as well."""
    N, C, H, W = x.shape
    O, C2, R, S = w.shape
    if C != C2 or x.dtype != torch.float32 or w.dtype != torch.float32:
        raise ValueError("float32 tensors with matching channels expected")
    P, Q = (H - 1) // 2 + 1, (W - 1) // 2 + 1
    if out.numel() != packed_act_words(N, O, (P - 1) // 2 + 1, (Q - 1) // 2 + 1, a_bits):
        raise ValueError("output of another size")
    st = lib().bs_stem_codes_operands_f32(_ptr(x), _ptr(w), _ptr(bias), N, C, H, W, O, R, S, 2, 3, act_scale, a_bits, _ptr(out), operands, _stream_ptr(stream))
    if st == ERR_UNSUPPORTED:
        return False
    _check(st, "bs_stem_codes_f32")
    return True


def stem_codes_supported(x_shape, w_shape, act_scale: float, a_bits: int) -> bool:
    """Whether :func:`stem_codes_f32` takes images and filters of these shapes."""
    N, C, H, W = x_shape
    O, C2, R, S = w_shape
    return C == C2 and bool(lib().bs_stem_codes_supported(N, C, H, W, O, R, S, 2, 3, act_scale, a_bits))


def avgpool_codes_f32(packed: torch.Tensor, C: int, a_sign: int, inv: float, out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """Global average pool of packed codes [N,H,W,Cw,a_bits] -> float32 [N,C] (``bs_avgpool_codes_f32``)."""
    N, H, W, Cw, a_bits = packed.shape
    if out is None:
        out = torch.empty(N, C, dtype=torch.float32, device=packed.device)
    _check(lib().bs_avgpool_codes_f32(_ptr(packed), N, C, H, W, a_bits, a_sign, ctypes.c_float(inv), _ptr(out), _stream_ptr(stream)),
           "bs_avgpool_codes_f32")
    return out


def fc_f32(x: torch.Tensor, w: torch.Tensor, bias: Optional[torch.Tensor] = None, out: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    N, K = x.shape
    J, K2 = w.shape
    if K != K2:
        raise ValueError("inner dimensions disagree")
    if out is None:
        out = torch.empty(N, J, dtype=torch.float32, device=x.device)
    _check(lib().bs_fc_f32(_ptr(x), _ptr(w), _ptr(bias), N, K, J, _ptr(out), _stream_ptr(stream)), "bs_fc_f32")
    return out


def bs_check_status(stream=None) -> None:
    st = lib().bs_check_status(_stream_ptr(stream))
    if st != 0:
        raise BitserialError(st, "bs_check_status")


def selftest_wait_timeout(polls: int = 256, stream=None) -> None:
    """Launches the kernel whose bounded wait runs out (``bs_selftest_wait_timeout``); the next :func:`bs_check_status`
    raises ``BitserialError`` with BS_ERR_TIMEOUT once."""
    _check(lib().bs_selftest_wait_timeout(int(polls), _stream_ptr(stream)), "bs_selftest_wait_timeout")


def l2_prefetch(tensors, stream=None) -> None:
    """Hint: bring the given device tensors into L2 while the following kernels of the stream run (``bs_l2_prefetch``)."""
    ts = [t for t in tensors if t is not None and t.numel() > 0]
    if not ts:
        return
    ptrs = (ctypes.c_void_p * len(ts))(*[t.data_ptr() for t in ts])
    sizes = (ctypes.c_size_t * len(ts))(*[t.numel() * t.element_size() for t in ts])
    _check(lib().bs_l2_prefetch(ptrs, sizes, len(ts), _stream_ptr(stream)), "bs_l2_prefetch")


def bs_popc_rate(iters: int = 4096) -> float:
    out = ctypes.c_double(0.0)
    st = lib().bs_popc_rate(iters, ctypes.byref(out))
    if st != 0:
        raise BitserialError(st, "bs_popc_rate")
    return out.value
