"""Thin ctypes binding over the three-dimensional entry points of libtconv.so (include/tconv3d.h).

Argument marshalling only; every step runs in the library's CUDA kernels.  A layer is described
by a dict with N, C, D, H, W, K, T, R, S, the triples ``stride`` / ``pad`` / ``dil`` in
(depth, height, width) order, and ``mode`` / ``chan`` / ``dtype`` by name.
"""
from __future__ import annotations

import ctypes

import torch

from .tconv import (CHANS, DTYPES, MODES, TORCH_DTYPE, KeptPlans, TconvError, _check, _lib, _on_stream, _p,
                    _ptr, _raw_stream, _stream)

# every symbol include/tconv3d.h declares
SYMBOLS = ("tconv3d_output_shape", "tconv3d_winner_bytes", "tconv3d_workspace_bytes", "tconv3d_forward",
           "tconv3d_backward", "tconv3d_launch_count")


class Desc3(ctypes.Structure):
    """tconv3d_desc_t."""
    _fields_ = [(n, ctypes.c_int32) for n in (
        "N", "C", "D", "H", "W", "K", "T", "R", "S", "stride_d", "stride_h", "stride_w", "pad_d", "pad_h",
        "pad_w", "dil_d", "dil_h", "dil_w", "mode", "chan", "dtype")]


def _bind():
    vp, fp, sz = ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t
    dp, ip = ctypes.POINTER(Desc3), ctypes.POINTER(ctypes.c_int32)
    _lib.tconv3d_output_shape.argtypes = [dp, ip, ip, ip]
    _lib.tconv3d_output_shape.restype = ctypes.c_int
    _lib.tconv3d_winner_bytes.argtypes = [dp]
    _lib.tconv3d_winner_bytes.restype = sz
    _lib.tconv3d_workspace_bytes.argtypes = [dp, ctypes.c_int]
    _lib.tconv3d_workspace_bytes.restype = sz
    _lib.tconv3d_forward.argtypes = [dp, vp, vp, vp, fp, fp, fp, vp, vp, vp]
    _lib.tconv3d_forward.restype = ctypes.c_int
    _lib.tconv3d_backward.argtypes = [dp, vp, vp, vp, fp, fp, vp, vp, vp, fp, fp, fp, fp, fp, vp, sz, vp]
    _lib.tconv3d_backward.restype = ctypes.c_int
    _lib.tconv3d_launch_count.restype = ctypes.c_longlong


_bind()


def make_desc(d: dict) -> Desc3:
    return Desc3(*(d[k] for k in "NCDHWKTRS"), *d["stride"], *d["pad"], *d["dil"], MODES[d["mode"]],
                 CHANS[d.get("chan", "default")], DTYPES[d.get("dtype", "f32")])


# ---- the C entry points, one to one ------------------------------------------------
def tconv3d_output_shape(d: dict):
    od, oh, ow = ctypes.c_int32(), ctypes.c_int32(), ctypes.c_int32()
    rc = _lib.tconv3d_output_shape(ctypes.byref(make_desc(d)), ctypes.byref(od), ctypes.byref(oh),
                                   ctypes.byref(ow))
    if rc != 0:
        raise TconvError(rc, "tconv3d_output_shape")
    return od.value, oh.value, ow.value


def tconv3d_winner_bytes(d: dict) -> int:
    return int(_lib.tconv3d_winner_bytes(ctypes.byref(make_desc(d))))


def tconv3d_workspace_bytes(d: dict, backward: bool) -> int:
    return int(_lib.tconv3d_workspace_bytes(ctypes.byref(make_desc(d)), int(backward)))


def tconv3d_forward(d: dict, x, w, w2, alpha, beta, bias, y, winners=None, stream=None) -> int:
    return _lib.tconv3d_forward(ctypes.byref(make_desc(d)), _p(x), _p(w), _p(w2), _p(alpha), _p(beta),
                                _p(bias), _p(y), _p(winners), _stream(stream))


def tconv3d_backward(d: dict, x, w, w2, alpha, beta, grad_y, winners, grad_x, grad_w, grad_w2, grad_alpha,
                     grad_beta, grad_bias, workspace, stream=None) -> int:
    nbytes = 0 if workspace is None else workspace.numel() * workspace.element_size()
    return _lib.tconv3d_backward(ctypes.byref(make_desc(d)), _p(x), _p(w), _p(w2), _p(alpha), _p(beta),
                                 _p(grad_y), _p(winners), _p(grad_x), _p(grad_w), _p(grad_w2),
                                 _p(grad_alpha), _p(grad_beta), _p(grad_bias), _p(workspace), nbytes,
                                 _stream(stream))


def tconv3d_launch_count() -> int:
    return int(_lib.tconv3d_launch_count())


# ---- allocation helpers -------------------------------------------------------------
def _shapes(d):
    N, C, D, H, W, K, T, R, S = (d[k] for k in "NCDHWKTRS")
    return (N, C, D, H, W), (K, C, T, R, S), (N, K) + tconv3d_output_shape(d)


class Plan3:
    """What a layer's calls need beside its tensors (see tconv.Plan)."""

    __slots__ = ("desc", "ref", "x", "w", "y", "kc", "k", "dt", "two", "par", "winner_shape", "winner_dtype", "bwd_ws")

    def __init__(self, d: dict):
        self.desc = make_desc(d)
        self.ref = ctypes.byref(self.desc)
        self.x, self.w, self.y = _shapes(d)
        self.kc, self.k = (d["K"], d["C"]), (d["K"],)
        self.dt = TORCH_DTYPE[d.get("dtype", "f32")]
        self.two, self.par = d["mode"] in ("compound", "parallel"), d["mode"] == "parallel"
        chan = d.get("chan", "default")
        if chan == "default":
            chan = {"max_plus": "max", "min_plus": "min"}.get(d["mode"], "sum")
        if chan == "sum":
            self.winner_shape, self.winner_dtype = self.y[:2] + (d["C"],) + self.y[2:], torch.int16
        else:
            self.winner_shape, self.winner_dtype = self.y, torch.int32
        self.bwd_ws = int(_lib.tconv3d_workspace_bytes(self.ref, 1))


_plans = KeptPlans(Plan3)
_FIELDS = ("N", "C", "D", "H", "W", "K", "T", "R", "S", "stride", "pad", "dil", "mode", "chan", "dtype")


def plan_of(d: dict) -> Plan3:
    return _plans.get(tuple(tuple(v) if isinstance(v, list) else v for v in map(d.get, _FIELDS)), d)


def winner_buffer(d: dict, device):
    """Buffer for the winning taps: uint16 [N,K,C,OD,OH,OW] (Sum channel combine) or int32 [N,K,OD,OH,OW]."""
    p = plan_of(d)
    return torch.empty(p.winner_shape, dtype=p.winner_dtype, device=device)


def forward(d: dict, x, w, w2=None, alpha=None, beta=None, bias=None, want_winners=False, stream=None):
    """Allocate y (and the winners) and run tconv3d_forward.  Returns (y, winners)."""
    p = plan_of(d)
    _check(x, p.x, p.dt, "x"); _check(w, p.w, p.dt, "w"); _check(w2, p.w, p.dt, "w2")
    _check(alpha, p.kc, torch.float32, "alpha"); _check(beta, p.kc, torch.float32, "beta")
    _check(bias, p.k, torch.float32, "bias")
    dev = x.device
    y = torch.empty(p.y, dtype=p.dt, device=dev)
    winners = torch.empty(p.winner_shape, dtype=p.winner_dtype, device=dev) if want_winners else None
    _on_stream(stream, y, winners)
    rc = _lib.tconv3d_forward(p.ref, x.data_ptr(), w.data_ptr(), _ptr(w2), _ptr(alpha), _ptr(beta), _ptr(bias),
                              y.data_ptr(), _ptr(winners), _raw_stream(stream))
    if rc != 0:
        raise TconvError(rc, "tconv3d_forward")
    return y, winners


def backward(d: dict, x, w, grad_y, w2=None, alpha=None, beta=None, winners=None, need_grad_x=True,
             stream=None):
    """Allocate every gradient the mode has and run tconv3d_backward.  Returns a dict."""
    p = plan_of(d)
    _check(x, p.x, p.dt, "x"); _check(w, p.w, p.dt, "w"); _check(w2, p.w, p.dt, "w2"); _check(grad_y, p.y, p.dt, "grad_y")
    dev, f32 = x.device, torch.float32
    out = {"grad_w": torch.empty(p.w, dtype=f32, device=dev), "grad_bias": torch.empty(p.k, dtype=f32, device=dev)}
    if need_grad_x:
        out["grad_x"] = torch.empty(p.x, dtype=p.dt, device=dev)
    if p.par:
        out["grad_w2"] = torch.empty(p.w, dtype=f32, device=dev)
    if p.two:
        out["grad_alpha"] = torch.empty(p.kc, dtype=f32, device=dev)
        out["grad_beta"] = torch.empty(p.kc, dtype=f32, device=dev)
    ws = torch.empty(p.bwd_ws, dtype=torch.uint8, device=dev)
    _on_stream(stream, ws, *out.values())
    get = out.get
    rc = _lib.tconv3d_backward(p.ref, x.data_ptr(), w.data_ptr(), _ptr(w2), _ptr(alpha), _ptr(beta),
                               grad_y.data_ptr(), _ptr(winners), _ptr(get("grad_x")), out["grad_w"].data_ptr(),
                               _ptr(get("grad_w2")), _ptr(get("grad_alpha")), _ptr(get("grad_beta")),
                               out["grad_bias"].data_ptr(), ws.data_ptr(), p.bwd_ws, _raw_stream(stream))
    if rc != 0:
        raise TconvError(rc, "tconv3d_backward")
    return out
