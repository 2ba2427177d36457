"""Python binding over libpf.so: argument marshalling only.

Every function has the name and the semantics of the C entry point it wraps (see
``include/pf.h``).  Tensors are torch CUDA tensors; torch is used for device memory and the
current stream, nothing else.  Outputs and workspaces that the caller does not pass come from
torch's caching allocator (the C library itself never allocates).  The marshalling is native
(``csrc/pf_python.cpp``, module ``_pf_native``): the functions here only give it names and
defaults.  ``lib()`` is the C library itself through ctypes.
"""
from __future__ import annotations

import ctypes
import os

import torch

PF_F32, PF_BF16 = 0, 1
PF_ACT_NONE, PF_ACT_RELU = 0, 1
PF_GRAD_ACCUMULATE, PF_GRAD_F32 = 1, 2
_PKG = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_PKG, "libpf.so")
_lib = None
_native = None


class PfError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {pf_status_string(status)} ({status})")


def lib() -> ctypes.CDLL:
    """The loaded C library; raises if it has not been built (no fallback path exists)."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise ImportError(
                f"{_LIB_PATH} is missing: build it with `python -m paper_2103_03936_b200.build` "
                "(there is no CPU or PyTorch fallback)")
        L = ctypes.CDLL(_LIB_PATH)
        i64, vp, sz, ci = ctypes.c_int64, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
        L.pf_status_string.restype = ctypes.c_char_p
        L.pf_status_string.argtypes = [ci]
        L.pf_version.restype = ci
        L.pf_last_device_status.restype = ci
        L.pf_launch_count.restype = ctypes.c_longlong
        L.pf_lowrank_linear_workspace.restype = sz
        L.pf_lowrank_linear_workspace.argtypes = [i64, i64, i64, i64, ci, ci]
        L.pf_lowrank_linear_fwd.restype = ci
        L.pf_lowrank_linear_fwd.argtypes = [vp, i64, vp, i64, vp, i64, vp, i64, vp, i64,
                                            i64, i64, i64, i64, ci, vp, sz, vp]
        L.pf_lowrank_linear_fwd_act.restype = ci
        L.pf_lowrank_linear_fwd_act.argtypes = [vp, i64, vp, i64, vp, i64, vp, ci, vp, i64, vp, i64,
                                                i64, i64, i64, i64, ci, vp, sz, vp]
        L.pf_bias_act_bwd_workspace.restype = sz
        L.pf_bias_act_bwd_workspace.argtypes = [i64, i64]
        L.pf_bias_act_bwd.restype = ci
        L.pf_bias_act_bwd.argtypes = [vp, i64, vp, i64, vp, i64, i64, ci, ci, vp, sz, vp]
        L.pf_lowrank_linear_fwd_static.restype = ci
        L.pf_lowrank_linear_fwd_static.argtypes = [vp, i64, vp, i64, vp, i64, vp, i64, vp, i64,
                                                   i64, i64, i64, i64, ci, vp]
        L.pf_static_scratch_bytes.restype = sz
        L.pf_lowrank_linear_bwd.restype = ci
        L.pf_lowrank_linear_bwd.argtypes = [vp, i64, vp, i64, vp, i64, vp, i64, vp, i64,
                                            vp, i64, vp, i64, vp, i64,
                                            i64, i64, i64, i64, ci, vp, sz, vp]
        L.pf_lowrank_linear_bwd_ex.restype = ci
        L.pf_lowrank_linear_bwd_ex.argtypes = [vp, i64, vp, i64, vp, i64, vp, i64, vp, i64,
                                               vp, i64, vp, i64, vp, i64, i64, i64, i64, i64, ci, ctypes.c_uint, vp, sz, vp]
        L.pf_lowrank_linear_grouped_workspace.restype = sz
        L.pf_lowrank_linear_grouped_workspace.argtypes = [ci, i64, i64, i64, i64, ci, ci]
        L.pf_lowrank_linear_grouped_fwd.restype = ci
        L.pf_lowrank_linear_grouped_fwd.argtypes = [ci] + [vp, i64, i64] * 5 + [i64, i64, i64, i64, ci, vp, sz, vp]
        L.pf_lowrank_linear_grouped_bwd.restype = ci
        L.pf_lowrank_linear_grouped_bwd.argtypes = [ci] + [vp, i64, i64] * 8 + [i64, i64, i64, i64, ci, vp, sz, vp]
        L.pf_lowrank_conv_workspace.restype = sz
        L.pf_lowrank_conv_workspace.argtypes = [ci] * 12
        L.pf_lowrank_conv_fwd.restype = ci
        L.pf_lowrank_conv_fwd.argtypes = [vp] * 5 + [ci] * 11 + [vp, sz, vp]
        L.pf_lowrank_conv_bwd.restype = ci
        L.pf_lowrank_conv_bwd.argtypes = [vp] * 8 + [ci] * 11 + [vp, sz, vp]
        L.pf_lowrank_conv_bwd_ex.restype = ci
        L.pf_lowrank_conv_bwd_ex.argtypes = [vp] * 8 + [ci] * 11 + [ctypes.c_uint, vp, sz, vp]
        L.pf_pack_factor_grads.restype = ci
        L.pf_pack_factor_grads.argtypes = [vp, vp, ci, ci, vp, i64, vp, vp, sz, vp]
        L.pf_unpack_factor_grads.restype = ci
        L.pf_unpack_factor_grads.argtypes = [vp, i64, vp, vp, ci, ci, vp, vp, sz, vp]
        _lib = L
    return _lib


def _load_native():
    """The marshalling module; raises if it has not been built."""
    global _native
    lib()
    path = os.path.join(_PKG, "_pf_native.so")
    if not os.path.exists(path):
        raise ImportError(f"{path} is missing: build it with `python -m paper_2103_03936_b200.build`")
    from . import _pf_native
    _pf_native.set_error(PfError)
    _native = _pf_native
    return _native


def pf_status_string(status: int) -> str:
    return lib().pf_status_string(int(status)).decode()


def pf_version() -> int:
    return int(lib().pf_version())


def pf_launch_count() -> int:
    return int(lib().pf_launch_count())


def pf_last_device_status() -> int:
    return int(lib().pf_last_device_status())


def pf_lowrank_linear_workspace(m, k, n, r, dtype, is_bwd) -> int:
    return int(lib().pf_lowrank_linear_workspace(m, k, n, r, dtype, int(bool(is_bwd))))


def pf_lowrank_linear_fwd(x, U, V, *, y=None, T_stash=None, want_stash=False, workspace=None,
                          stream=None, prepare=False):
    """y = (x U) V^T.  Returns y, or (y, T_stash) when a stash is requested.
    With prepare=True nothing is launched: returns (call, outputs) where call() issues the
    C call with the arguments marshalled once (fixed buffers and stream)."""
    n = _native or _load_native()
    return n.linear_fwd(x, U, V, None, 0, y, T_stash, want_stash, workspace, stream, prepare, False)


def pf_lowrank_linear_fwd_act(x, U, V, *, bias=None, act=PF_ACT_NONE, y=None, T_stash=None, want_stash=False,
                              workspace=None, stream=None, prepare=False):
    """y = act((x U) V^T + bias); bias [n] in x's dtype or None, act PF_ACT_NONE / PF_ACT_RELU.
    Otherwise as pf_lowrank_linear_fwd."""
    n = _native or _load_native()
    return n.linear_fwd(x, U, V, bias, act, y, T_stash, want_stash, workspace, stream, prepare, True)


def pf_bias_act_bwd(y, dY, *, act=PF_ACT_RELU, want_dbias=True, dbias=None, workspace=None, stream=None):
    """Backward of y = act(z + bias): dY [m, n] becomes dZ IN PLACE (zeroed where y <= 0 for PF_ACT_RELU);
    returns dbias [n] (column sums of dZ) or None."""
    n = _native or _load_native()
    return n.bias_act_bwd(y, dY, act, want_dbias, dbias, workspace, stream)


def pf_static_scratch_bytes() -> int:
    return int(lib().pf_static_scratch_bytes())


def pf_lowrank_linear_fwd_static(x, U, V, *, y, T_stash=None, stream=None):
    """y = (x U) V^T for callers that cannot allocate: the scratch is a fixed array inside the
    library, so the caller passes inputs and outputs only (y is required; nothing is allocated
    here either).  Raises PfError(PF_ERR_WORKSPACE) when the problem does not fit the array.
    Calls on one device share that array: do not let two of them overlap on the GPU."""
    n = _native or _load_native()
    return n.linear_fwd_static(x, U, V, y, T_stash, stream)


def pf_lowrank_linear_bwd(x, U, V, dY, *, T_stash=None, need_dX=True, dX=None, dU=None, dV=None,
                          accumulate=False, grads_f32=False, workspace=None, stream=None, prepare=False):
    """Returns (dX or None, dU, dV) for upstream gradient dY (prepare: see the forward).
    accumulate: dU and dV (required then) are added to; grads_f32: dU and dV are fp32 tensors."""
    n = _native or _load_native()
    return n.linear_bwd(x, U, V, dY, T_stash, need_dX, dX, dU, dV, accumulate, grads_f32, workspace, stream, prepare)


def pf_lowrank_linear_grouped_workspace(groups, m, k, n, r, dtype, is_bwd) -> int:
    return int(lib().pf_lowrank_linear_grouped_workspace(groups, m, k, n, r, dtype, int(bool(is_bwd))))


def pf_lowrank_linear_grouped_fwd(x, U, V, *, y=None, T_stash=None, want_stash=False, workspace=None,
                                  stream=None, prepare=False):
    """y[g] = (x[g] U[g]) V[g]^T for U [G, k, r], V [G, n, r] and x [G, m, k] or one shared x [m, k].
    Returns y [G, m, n], or (y, T_stash [G, m, r]) when a stash is requested."""
    n = _native or _load_native()
    return n.grouped_fwd(x, U, V, y, T_stash, want_stash, workspace, stream, prepare)


def pf_lowrank_linear_grouped_bwd(x, U, V, dY, *, T_stash=None, need_dX=True, dX=None, dU=None, dV=None,
                                  workspace=None, stream=None, prepare=False):
    """Returns (dX or None, dU [G, k, r], dV [G, n, r]).  dX is [G, m, k] when every group has its own
    x and ONE [m, k] matrix (the sum over the groups) when x [m, k] is shared."""
    n = _native or _load_native()
    return n.grouped_bwd(x, U, V, dY, T_stash, need_dX, dX, dU, dV, workspace, stream, prepare)


def pf_lowrank_conv_workspace(N, H, W, C, R, O, kh, kw, stride, pad, dtype, is_bwd) -> int:
    return int(lib().pf_lowrank_conv_workspace(N, H, W, C, R, O, kh, kw, stride, pad, dtype,
                                               int(bool(is_bwd))))


def pf_lowrank_conv_fwd(x, U, V, *, stride=1, pad=1, y=None, T_stash=None, want_stash=False,
                        workspace=None, stream=None, prepare=False):
    """NHWC factorized convolution.  Returns y, or (y, T_stash) when a stash is requested."""
    n = _native or _load_native()
    return n.conv_fwd(x, U, V, stride, pad, y, T_stash, want_stash, workspace, stream, prepare)


def pf_lowrank_conv_bwd(x, U, V, dY, *, stride=1, pad=1, T_stash=None, need_dX=True, dX=None,
                        dU=None, dV=None, accumulate=False, grads_f32=False, workspace=None, stream=None,
                        prepare=False):
    """Returns (dX or None, dU, dV) for upstream gradient dY [N, Ho, Wo, O].
    accumulate / grads_f32: as in pf_lowrank_linear_bwd."""
    n = _native or _load_native()
    return n.conv_bwd(x, U, V, dY, stride, pad, T_stash, need_dX, dX, dU, dV, accumulate, grads_f32, workspace, stream,
                      prepare)


def pf_pack_factor_grads(grads, *, flat=None, stream=None, prepare=False):
    """Copies the tensors of `grads`, in order and tightly, into one flat buffer.
    Returns (flat, offsets) with offsets a python list of count+1 element offsets."""
    if len(grads) == 0:
        offs = (ctypes.c_int64 * 1)()
        st = lib().pf_pack_factor_grads(None, None, 0, PF_BF16, flat.data_ptr() if flat is not None else None,
                                        flat.numel() if flat is not None else 0, offs, None, 0, None)
        if st != 0:
            raise PfError(st, "pf_pack_factor_grads")
        return flat, [0]
    n = _native or _load_native()
    return n.pack(grads, flat, stream, prepare)


def pf_unpack_factor_grads(flat, grads, *, stream=None):
    """The inverse of pf_pack_factor_grads: tensor i of `grads` (contiguous CUDA tensors of flat's
    dtype, overwritten) receives its slice of `flat`.  Returns the list of count+1 element offsets."""
    if len(grads) == 0:
        return [0]
    n = _native or _load_native()
    return n.unpack(flat, grads, stream)
