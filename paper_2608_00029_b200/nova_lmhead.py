"""Binding of the loss-head entry points of libnova_attn.so (include/nova_lmhead.h): same names as the
C ABI, argument checks and marshalling only.  No CPU fallback: a missing library or a failed call raises."""
from __future__ import annotations

import ctypes

from . import nova_attn as _na

_ready = False


def _lib():
    global _ready
    lib = _na.load()
    if not _ready:
        vp, i, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t
        lib.nova_lmhead_workspace_bytes.argtypes = [i, i, i]
        lib.nova_lmhead_workspace_bytes.restype = sz
        lib.nova_lmhead_fwd.argtypes = [vp] * 6 + [i, i, i, vp, sz, vp]
        lib.nova_lmhead_fwd.restype = i
        _ready = True
    return lib


def nova_lmhead_workspace_bytes(M: int, N: int, K: int) -> int:
    return int(_lib().nova_lmhead_workspace_bytes(M, N, K))


def nova_lmhead_fwd(X, W, targets, logits, lse, loss, workspace=None, stream=None) -> None:
    """lse, loss (and logits unless None) <- loss head of X [M,K] against W [N,K] with int32 targets [M].
    X, W, logits are contiguous CUDA bf16 tensors, targets, lse and loss contiguous [M]; `workspace` is a
    CUDA tensor without gaps of at least nova_lmhead_workspace_bytes(M, N, K) bytes (allocated here if omitted)."""
    rc = _na._binding().lmhead_fwd(X, W, targets, logits, lse, loss, workspace, stream)
    if rc != _na.OK:
        raise _na.NovaAttnError(rc, "nova_lmhead_fwd")
