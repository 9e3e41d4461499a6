"""Python binding of the rmuscle C-ABI library (activation-masked gated MLP of an action expert on B200).

The binding only marshals arguments: every tensor is a torch CUDA tensor whose data pointer is handed to the
`extern "C"` entry point of the same name, on torch's current stream.  The calls of a control loop go through a small
CPython module (csrc/rm_python.cpp: a call's marshalling through ctypes took longer on the host than the shorter kernels
take on the GPU), set-up and diagnostics through ctypes.  There is no CPU path: loading fails with an error when the CUDA
library has not been built (`python -m paper_2609_19104_b200.build`).
"""
from __future__ import annotations

import ctypes
import importlib.machinery
import importlib.util
import os
from typing import Optional, Sequence

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "librmuscle.so")
MODULE_PATH = os.path.join(_PKG, "_rmuscle.so")

RM_OK = 0
RM_ERR_INVALID_ARG, RM_ERR_SHAPE, RM_ERR_ALIGN, RM_ERR_WORKSPACE = -1, -2, -3, -4
RM_ERR_CUDA, RM_ERR_INDEX, RM_ERR_TIMEOUT, RM_ERR_UNSUPPORTED = -5, -6, -7, -8
RM_ACT_GELU_TANH = 0
RM_SRC_BOOL_U8, RM_SRC_SCORE_F32 = 0, 1
RM_REDUCE_NONE, RM_REDUCE_THRESHOLD, RM_REDUCE_TOPK, RM_REDUCE_GROUP = 0, 1, 2, 3
RM_ANCHOR_NONE, RM_ANCHOR_WRITE, RM_ANCHOR_UPDATE = 0, 1, 2

EXPORTS = ["rm_create", "rm_destroy", "rm_packed_layer_bytes", "rm_workspace_bytes", "rm_pack_weights",
           "rm_mask_compact", "rm_sparse_mlp", "rm_action_expert_step", "rm_action_expert_step_host",
           "rm_action_expert_step_ex", "rm_gather_weights", "rm_context_drift", "rm_context_workspace_bytes",
           "rm_context_ffn", "rm_debug_gather_read", "rm_debug_gather_read_step", "rm_debug_wait_timeout",
           "rm_device_status", "rm_launch_count", "rm_status_string", "rm_set_option", "rm_get_info",
           "rm_debug_phase_times", "rm_sparse_mlp_static"]


class RmError(RuntimeError):
    def __init__(self, code: int, where: str):
        self.code = code
        extra = ""
        if code == -5 and _lib is not None:                # RM_ERR_CUDA: add the runtime's own error code
            v = ctypes.c_int(0)
            if _lib.rm_get_info(None, b"last_cuda_error", ctypes.byref(v)) == 0:
                extra = f" [cudaError_t {v.value}]"
        super().__init__(f"{where}: {status_string(code)} ({code}){extra}")


class rm_model_desc(ctypes.Structure):
    _fields_ = [("L", ctypes.c_int32), ("H", ctypes.c_int32), ("I", ctypes.c_int32), ("T_max", ctypes.c_int32),
                ("B_max", ctypes.c_int32), ("act", ctypes.c_int32)]


class rm_mask_src(ctypes.Structure):
    _fields_ = [("kind", ctypes.c_int32), ("reduce", ctypes.c_int32), ("threshold", ctypes.c_float),
                ("k", ctypes.c_int32), ("n_records", ctypes.c_int32), ("min_votes", ctypes.c_int32),
                ("records", ctypes.POINTER(ctypes.c_void_p)), ("scale", ctypes.c_void_p),
                ("scale_per_list", ctypes.c_int32), ("n_lists", ctypes.c_int32), ("I", ctypes.c_int32)]


_lib = None
_native = None


def load_library() -> ctypes.CDLL:
    """Loads librmuscle.so; raises when it is missing (there is no fallback path)."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise ImportError(f"{LIB_PATH} is missing: build it with `python -m paper_2609_19104_b200.build` "
                          "(nvcc, sm_100a); this package has no CPU or PyTorch fallback")
    lib = ctypes.CDLL(LIB_PATH)
    vp, i32, i64, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64, ctypes.c_size_t
    lib.rm_create.argtypes = [ctypes.POINTER(vp), ctypes.POINTER(rm_model_desc)]
    lib.rm_destroy.argtypes = [vp]
    lib.rm_packed_layer_bytes.argtypes = [vp]
    lib.rm_packed_layer_bytes.restype = sz
    lib.rm_workspace_bytes.argtypes = [vp, i32, i32]
    lib.rm_workspace_bytes.restype = sz
    lib.rm_pack_weights.argtypes = [vp, vp, vp, vp, vp, vp, vp]
    lib.rm_mask_compact.argtypes = [vp, ctypes.POINTER(rm_mask_src), vp, vp, i64, vp]
    lib.rm_sparse_mlp.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, vp, i32, vp, sz, vp]
    lib.rm_action_expert_step.argtypes = [vp, ctypes.POINTER(vp), vp, vp, vp, i64, vp, vp, vp, i32, i32, vp, sz, vp]
    lib.rm_action_expert_step_host.argtypes = [vp, ctypes.POINTER(vp), vp, vp, vp, i64, vp, i32, i32, vp, sz, vp]
    lib.rm_context_drift.argtypes = [vp, vp, vp, i32, vp, vp]
    lib.rm_context_workspace_bytes.argtypes = [vp, i32]
    lib.rm_context_workspace_bytes.restype = sz
    lib.rm_context_ffn.argtypes = [vp, vp, vp, vp, vp, vp, vp, i32, i32, i32, vp, vp, vp, sz, vp]
    lib.rm_debug_gather_read.argtypes = [vp, vp, vp, vp, i64, vp]
    lib.rm_gather_weights.argtypes = [vp, vp, vp, vp, i64, vp, vp]
    lib.rm_debug_gather_read_step.argtypes = [vp, ctypes.POINTER(vp), vp, vp, i64, vp]
    lib.rm_debug_wait_timeout.argtypes = [vp, i32, vp]
    lib.rm_action_expert_step_ex.argtypes = [vp, ctypes.POINTER(vp), vp, vp, vp, i64, vp, vp, vp, i32, i32, i32, vp, vp,
                                             i64, vp, vp, sz, vp]
    lib.rm_device_status.argtypes = [vp, ctypes.POINTER(ctypes.c_int), vp]
    lib.rm_launch_count.argtypes = [vp]
    lib.rm_launch_count.restype = i64
    lib.rm_set_option.argtypes = [vp, ctypes.c_char_p, i32]
    lib.rm_get_info.argtypes = [vp, ctypes.c_char_p, ctypes.POINTER(ctypes.c_int)]
    lib.rm_debug_phase_times.argtypes = [vp, ctypes.POINTER(ctypes.c_longlong), i32]
    lib.rm_sparse_mlp_static.argtypes = [vp, vp, vp, vp, vp, vp, i32, i32, i32, vp]
    lib.rm_status_string.argtypes = [i32]
    lib.rm_status_string.restype = ctypes.c_char_p
    for name in EXPORTS:
        getattr(lib, name)
    _load_module()
    _lib = lib
    return lib


def _load_module() -> None:
    """Loads the CPython module next to the library (it links against that same file)."""
    global _native
    if not os.path.exists(MODULE_PATH):
        raise ImportError(f"{MODULE_PATH} is missing: build it with `python -m paper_2609_19104_b200.build`")
    import torch
    loader = importlib.machinery.ExtensionFileLoader("_rmuscle", MODULE_PATH)
    mod = importlib.util.module_from_spec(importlib.util.spec_from_file_location("_rmuscle", MODULE_PATH, loader=loader))
    loader.exec_module(mod)
    # (a torch without CUDA has neither; nothing but Context, which refuses to exist there, would call them)
    mod.init(getattr(torch._C, "_cuda_getDevice", None), getattr(torch._C, "_cuda_getCurrentRawStream", None))
    _native = mod


def status_string(code: int) -> str:
    return load_library().rm_status_string(int(code)).decode()


def _check(code: int, where: str) -> None:
    if code != RM_OK:
        raise RmError(code, where)


def _ptr(t) -> Optional[int]:
    return None if t is None else int(t.data_ptr())


def _stream() -> int:
    import torch
    return int(torch.cuda.current_stream().cuda_stream)


def rm_sparse_mlp_static(packed_layer, x, residual, idx, count_dev, y, T: int, H: int, I: int):
    """One masked MLP layer without a context, a workspace or any allocation: the scratch is a fixed array inside the
    library (T * I <= 1,048,576).  For callers that may not allocate device memory.  Calls that overlap on the GPU
    share that array and must be serialised; make the first call on a device outside stream capture."""
    load_library()
    _check(_native.sparse_mlp_static(packed_layer, x, residual, idx, count_dev, y, T, H, I), "rm_sparse_mlp_static")
    return y


class Context:
    """Owns an rm_ctx for one model geometry on the current CUDA device."""

    def __init__(self, L: int, H: int, I: int, T_max: int, B_max: int = 1):
        import torch
        if not torch.cuda.is_available():
            raise RuntimeError("rmuscle needs a CUDA device; there is no CPU path")
        self.lib = load_library()
        self.L, self.H, self.I, self.T_max, self.B_max = L, H, I, T_max, B_max
        desc = rm_model_desc(L, H, I, T_max, B_max, RM_ACT_GELU_TANH)
        self._h = ctypes.c_void_p()
        _check(self.lib.rm_create(ctypes.byref(self._h), ctypes.byref(desc)), "rm_create")
        self._hv = self._h.value
        self._ws = None
        self._ws_bytes = 0
        self._ws_need = {}                                         # (B, T) -> bytes; R_max -> bytes of the Context Cache
        self._ctx_ws, self._ctx_ws_bytes = None, 0

    def close(self) -> None:
        if getattr(self, "_h", None) is not None and self._h.value:
            self.lib.rm_destroy(self._h)
            self._h = ctypes.c_void_p()
            self._hv = 0

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    # ------------------------------------------------------------------ sizes
    def packed_layer_bytes(self) -> int:
        return int(self.lib.rm_packed_layer_bytes(self._h))

    def workspace_bytes(self, B: int, T: int) -> int:
        return int(self.lib.rm_workspace_bytes(self._h, B, T))

    def workspace(self, B: int, T: int):
        """A cached torch byte buffer large enough for (B, T)."""
        import torch
        need = self.workspace_bytes(B, T)
        if self._ws is None or self._ws.numel() < need:
            self._ws = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
            self._ws_bytes = self._ws.numel()
        return self._ws

    def _scratch(self, B: int, T: int, ws):
        """(workspace, its bytes) of a call: the caller's, or the cached one."""
        if ws is not None:
            return ws, ws.numel()
        key = (B, T)
        need = self._ws_need.get(key)
        if need is None:
            need = self._ws_need[key] = self.workspace_bytes(max(B, 1), max(T, 1))
        if self._ws is None or self._ws_bytes < need:
            self.workspace(max(B, 1), max(T, 1))
        return self._ws, self._ws_bytes

    def rm_set_option(self, name: str, value: int) -> None:
        _check(self.lib.rm_set_option(self._h, name.encode(), int(value)), f"rm_set_option({name})")

    def rm_get_info(self, name: str) -> int:
        v = ctypes.c_int(0)
        _check(self.lib.rm_get_info(self._h, name.encode(), ctypes.byref(v)), f"rm_get_info({name})")
        return int(v.value)

    def rm_debug_phase_times(self, n_ctas: int):
        """Clock stamps [n_ctas, 32] of the last fused-layer launch (builds with -DRM_PHASE_TIMING only)."""
        import numpy as np
        buf = (ctypes.c_longlong * (n_ctas * 32))()
        _check(self.lib.rm_debug_phase_times(self._h, buf, n_ctas * 32), "rm_debug_phase_times")
        return np.frombuffer(buf, dtype=np.int64).reshape(n_ctas, 32).copy()

    def launch_count(self) -> int:
        return int(self.lib.rm_launch_count(self._h))

    # ------------------------------------------------------------------ calls (same names as the C ABI)
    def rm_pack_weights(self, Wg, Wu, Wd, packed_out=None, down_colnorm=None):
        import torch
        if packed_out is None:
            packed_out = torch.empty(self.packed_layer_bytes(), dtype=torch.uint8, device="cuda")
        _check(self.lib.rm_pack_weights(self._h, _ptr(Wg), _ptr(Wu), _ptr(Wd), _ptr(packed_out), _ptr(down_colnorm),
                                        _stream()), "rm_pack_weights")
        return packed_out

    def rm_mask_compact(self, records: Sequence, kind: int, reduce: int, idx_out, count_out, stride: int, *,
                        n_lists: int, threshold: float = 0.0, k: int = 0, min_votes: int = 1, scale=None,
                        scale_per_list: bool = False, I: Optional[int] = None):
        rc = _native.mask_compact(self._hv, records, kind, reduce, threshold, k, min_votes, scale, scale_per_list, n_lists,
                                  self.I if I is None else I, idx_out, count_out, stride)
        if rc != RM_OK:
            raise RmError(rc, "rm_mask_compact")

    def rm_context_drift(self, x, x_ref, P: int, score_out):
        """Eq. 2: per-row drift score of the current FFN input against the reference input."""
        _check(_native.context_drift(self._hv, x, x_ref, P, score_out), "rm_context_drift")
        return score_out

    def rm_context_ffn(self, Wg, Wu, Wd, x, rows, count_dev, P: int, S: int, R_max: int, y_ref, y_out, ws=None):
        """Eq. 3: recompute the listed visual rows and the S always-recomputed rows, keep y_ref elsewhere."""
        if ws is None:
            need = self._ws_need.get(R_max)
            if need is None:
                need = self._ws_need[R_max] = int(self.lib.rm_context_workspace_bytes(self._h, int(R_max)))
            ws = self._ctx_ws
            if ws is None or self._ctx_ws_bytes < need:
                import torch
                ws = self._ctx_ws = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
                self._ctx_ws_bytes = ws.numel()
            ws_bytes = self._ctx_ws_bytes
        else:
            ws_bytes = ws.numel()
        _check(_native.context_ffn(self._hv, Wg, Wu, Wd, x, rows, count_dev, P, S, R_max, y_ref, y_out, ws, ws_bytes),
               "rm_context_ffn")
        return y_out

    def rm_debug_gather_read(self, packed_layer, idx, count_dev, list_cap: int):
        """Measurement aid: read the listed neurons' rows with the kernels' access pattern and discard them."""
        _check(self.lib.rm_debug_gather_read(self._h, _ptr(packed_layer), _ptr(idx), _ptr(count_dev), int(list_cap),
                                             _stream()), "rm_debug_gather_read")

    def rm_debug_gather_read_step(self, packed_layers, idx, count_dev, stride: int):
        """Measurement aid: the L lists of one episode's step read in one launch and discarded."""
        _check(self.lib.rm_debug_gather_read_step(self._h, self._layer_ptrs(packed_layers), _ptr(idx), _ptr(count_dev),
                                                  int(stride), _stream()), "rm_debug_gather_read_step")

    def rm_debug_wait_timeout(self, polls: int = 4096):
        """Test aid: one CTA whose bounded wait runs out (records RM_ERR_TIMEOUT and returns)."""
        _check(self.lib.rm_debug_wait_timeout(self._h, int(polls), _stream()), "rm_debug_wait_timeout")

    def rm_gather_weights(self, packed_layer, idx, count_dev, list_cap: int, compact_out=None):
        """Compact copy of the listed neurons' packed rows (a packed layer whose leading `count` neurons are the list)."""
        import torch
        if compact_out is None:
            compact_out = torch.empty(self.packed_layer_bytes(), dtype=torch.uint8, device="cuda")
        _check(self.lib.rm_gather_weights(self._h, _ptr(packed_layer), _ptr(idx), _ptr(count_dev), int(list_cap),
                                          _ptr(compact_out), _stream()), "rm_gather_weights")
        return compact_out

    def rm_sparse_mlp(self, packed_layer, x, residual, idx, count_dev, y, record_out=None, record_scale=None,
                      T: Optional[int] = None, ws=None):
        T = int(x.shape[0]) if T is None else T
        ws, ws_bytes = self._scratch(1, T, ws)
        _check(_native.sparse_mlp(self._hv, packed_layer, x, residual, idx, count_dev, y, record_out, record_scale, T, ws,
                                  ws_bytes), "rm_sparse_mlp")
        return y

    def _layer_ptrs(self, packed_layers):
        if len(packed_layers) < self.L:
            raise ValueError(f"{len(packed_layers)} packed layers for a model of {self.L}")
        return (ctypes.c_void_p * len(packed_layers))(*[_ptr(p) for p in packed_layers])

    def rm_action_expert_step(self, packed_layers, r_in, idx, count_dev, stride: int, r_out, records_out=None,
                              record_scale=None, B: int = 1, T: Optional[int] = None, ws=None):
        T = int(r_in.shape[-2]) if T is None else T
        ws, ws_bytes = self._scratch(B, T, ws)
        _check(_native.step(self._hv, packed_layers, self.L, r_in, idx, count_dev, stride, r_out, records_out, record_scale, B, T, ws,
                            ws_bytes), "rm_action_expert_step")
        return r_out

    def rm_action_expert_step_ex(self, packed_layers, r_in, idx, count_dev, stride: int, r_out, anchor_mode: int,
                                 y_anchor, h_anchor, h_stride: int, out_gate=None, records_out=None,
                                 record_scale=None, B: int = 1, T: Optional[int] = None, ws=None):
        """The step with the anchor-relative update (Eq. 4): y_anchor [L,B,T,H], h_anchor [L,B,I,h_stride] fp32."""
        T = int(r_in.shape[-2]) if T is None else T
        ws, ws_bytes = self._scratch(B, T, ws)
        _check(_native.step_ex(self._hv, packed_layers, self.L, r_in, idx, count_dev, stride, r_out, records_out, record_scale, B, T,
                               anchor_mode, y_anchor, h_anchor, h_stride, out_gate, ws, ws_bytes), "rm_action_expert_step_ex")
        return r_out

    def rm_action_expert_step_host(self, packed_layers, r_in_host, idx, count_dev, stride: int, r_out_host,
                                   B: int = 1, T: Optional[int] = None, ws=None):
        """r_in_host / r_out_host are CPU tensors (pinned for asynchronous copies); returns after the result landed."""
        T = int(r_in_host.shape[-2]) if T is None else T
        ws, ws_bytes = self._scratch(B, T, ws)
        _check(_native.step_host(self._hv, packed_layers, self.L, r_in_host, idx, count_dev, stride, r_out_host, B, T, ws, ws_bytes),
               "rm_action_expert_step_host")
        return r_out_host

    def rm_device_status(self) -> int:
        v = ctypes.c_int(0)
        _check(self.lib.rm_device_status(self._h, ctypes.byref(v), _stream()), "rm_device_status")
        return int(v.value)
