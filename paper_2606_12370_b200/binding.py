"""ctypes binding of libbebop.so.  Same names as the C ABI (include/bebop.h).

Argument marshalling only: tensors are torch CUDA tensors whose device pointers
are handed to the library, outputs are allocated when not supplied, and the
call is enqueued on torch's current stream.  Nothing is computed here: the four
calls go through the native marshaller csrc/bebop_host.cpp (_bebop_host.so, built
beside the library), everything else through ctypes.
"""
import ctypes as C
import importlib
import os

import torch

BEBOP_F32, BEBOP_BF16 = 0, 1
_HERE = os.path.dirname(os.path.abspath(__file__))
_LIB_PATH = os.path.join(_HERE, "libbebop.so")
_lib = None
_host = None


class BebopError(RuntimeError):
    def __init__(self, code: int, msg: str):
        super().__init__("bebop status %d: %s" % (code, msg))
        self.code = code


def library_path() -> str:
    return _LIB_PATH


def load_library():
    """Load libbebop.so (never builds, never falls back)."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(_LIB_PATH):
        raise ImportError("%s is missing: build it with `python -m paper_2606_12370_b200.build` "
                          "(there is no CPU fallback)" % _LIB_PATH)
    lib = C.CDLL(_LIB_PATH)
    vp, i64, i32, f32, sz = C.c_void_p, C.c_int64, C.c_int, C.c_float, C.c_size_t
    lib.bebop_workspace_bytes.restype = sz
    lib.bebop_workspace_bytes.argtypes = [i32, i32, i32, i32]
    lib.bebop_verify.restype = i32
    lib.bebop_verify.argtypes = [vp, i64, vp, i64, vp, vp, vp, f32, vp, vp, i32, i32, i32, i32,
                                 vp, vp, vp, vp, vp, vp, vp, sz, vp]
    lib.bebop_tv.restype = i32
    lib.bebop_tv.argtypes = [vp, i64, vp, i64, vp, f32, i32, i32, i32, vp, vp, vp, vp, sz, vp]
    lib.bebop_tv_static.restype = i32
    lib.bebop_tv_static.argtypes = [vp, i64, vp, i64, vp, f32, i32, i32, i32, vp, vp, vp, vp]
    lib.bebop_greedy_verify.restype = i32
    lib.bebop_greedy_verify.argtypes = [vp, i64, vp, vp, i32, i32, i32, i32, vp, vp, vp, vp, sz, vp]
    lib.bebop_debug_force_general_path.restype = None
    lib.bebop_debug_force_general_path.argtypes = [i32]
    lib.bebop_debug_set_timing_events.restype = None
    lib.bebop_debug_set_timing_events.argtypes = [vp, vp]
    lib.bebop_debug_last_kernel.restype = C.c_int
    lib.bebop_debug_last_kernel.argtypes = []
    lib.bebop_debug_last_kernel_name.restype = C.c_char_p
    lib.bebop_debug_last_kernel_name.argtypes = []
    lib.bebop_debug_set_draw_kappa.restype = None
    lib.bebop_debug_set_draw_kappa.argtypes = [f32]
    lib.bebop_debug_expire_wait.restype = None
    lib.bebop_debug_expire_wait.argtypes = [i32]
    lib.bebop_debug_fallback_offset.restype = sz
    lib.bebop_debug_fallback_offset.argtypes = [i32, i32, i32, i32]
    lib.bebop_status_string.restype = C.c_char_p
    lib.bebop_status_string.argtypes = [i32]
    _lib = lib
    return lib


def bebop_status_string(code: int) -> str:
    return load_library().bebop_status_string(int(code)).decode()


def _check(code: int):
    if code != 0:
        raise BebopError(code, bebop_status_string(code))


_HOST_CODES = {-8: (8, "tensors must live on a CUDA device (no CPU fallback)"),
               -3: (3, "logits must be float32 or bfloat16")}


def _load_host():
    """The native marshaller, bound to the library's entry points (never builds, never falls back)."""
    global _host
    lib = load_library()
    try:
        host = importlib.import_module("._bebop_host", __package__)
    except ImportError as e:
        raise ImportError("_bebop_host.so is missing or does not load: build it with "
                          "`python -m paper_2606_12370_b200.build`") from e
    host.init(*(C.cast(f, C.c_void_p).value for f in
                (lib.bebop_verify, lib.bebop_tv, lib.bebop_tv_static, lib.bebop_greedy_verify, lib.bebop_workspace_bytes)))
    _host = host
    return host


def _result(r):
    """The marshaller's answer: the outputs, or the code of what went wrong."""
    if type(r) is not int:
        return r
    if r in _HOST_CODES:
        raise BebopError(*_HOST_CODES[r])
    _check(r)


def bebop_debug_force_general_path(on) -> None:
    load_library().bebop_debug_force_general_path(int(on))


def bebop_debug_last_kernel() -> int:
    """What the last bebop_verify / bebop_tv / bebop_greedy_verify call ran: 1 general kernels, 2 pipelined kernel,
    3 a kernel that reads every logit once (fused or sequence kernel)."""
    return int(load_library().bebop_debug_last_kernel())


def bebop_debug_last_kernel_name() -> str:
    """The main kernel of the last of these calls: "general", "k_pipe", "k_fuse", "k_seq" or "k_seq_greedy" ("none": no call yet)."""
    return load_library().bebop_debug_last_kernel_name().decode()


def bebop_debug_set_draw_kappa(kappa) -> None:
    """Factor of the fast draw's error bound (built-in 4; negative restores it; 0 keeps every fp32 draw)."""
    load_library().bebop_debug_set_draw_kappa(float(kappa))


def bebop_debug_expire_wait(which) -> None:
    """The next call lets device-side wait `which` (1: re-draw list, 2: accept scan) give up at once; 0 = off."""
    load_library().bebop_debug_expire_wait(int(which))


def bebop_debug_set_timing_events(start, stop) -> None:
    """torch.cuda.Event pair (enable_timing=True, already recorded once) bracketing the main (pipelined) kernel; None, None = off."""
    lib = load_library()
    if start is None:
        lib.bebop_debug_set_timing_events(None, None)
    else:
        lib.bebop_debug_set_timing_events(C.c_void_p(start.cuda_event), C.c_void_p(stop.cuda_event))


def bebop_debug_fallback_offset(B: int, K: int, V: int, dt: int) -> int:
    return int(load_library().bebop_debug_fallback_offset(B, K, V, dt))


def bebop_workspace_bytes(B: int, K: int, V: int, dt: int) -> int:
    return int(load_library().bebop_workspace_bytes(B, K, V, dt))


# Tests set this so that an output the library failed to write cannot pass as a left-over of an
# earlier call in recycled memory.
POISON_OUTPUTS = False


def bebop_verify(target_logits, draft_logits, draft_tokens, u_accept, u_final, draft_len=None,
                 temperature=None, temperature_all=1.0, out=None, workspace=None,
                 want_tv=True, want_probs=True, want_status=True):
    """Chain rejection-sampling verification.  Returns a dict of CUDA tensors:
    accept_len [B] i32, out_tokens [B,K+1] i32, tv / p_draft / q_draft [B,K] f32,
    row_status [B] i32 (the optional ones are None when not requested)."""
    return _result((_host or _load_host()).verify(target_logits, draft_logits, draft_tokens, u_accept, u_final, draft_len, temperature,
                                                  temperature_all, None if not out else out if isinstance(out, dict) else dict(out), workspace, want_tv, want_probs, want_status, POISON_OUTPUTS))


def bebop_tv(target_logits, draft_logits, temperature=None, temperature_all=1.0, workspace=None,
             want_s_aux=True, want_status=True):
    """TV distance (and the auxiliary S) of N paired rows [N,V]."""
    return _result((_host or _load_host()).tv(target_logits, draft_logits, temperature, temperature_all, workspace, want_s_aux, want_status,
                                              POISON_OUTPUTS, False))


def bebop_tv_static(target_logits, draft_logits, temperature=None, temperature_all=1.0, want_s_aux=True):
    """bebop_tv with the library's built-in scratch instead of a workspace (no allocation in the call)."""
    return _result((_host or _load_host()).tv(target_logits, draft_logits, temperature, temperature_all, None, want_s_aux, True,
                                              POISON_OUTPUTS, True))


def bebop_greedy_verify(target_logits, draft_tokens, draft_len=None, workspace=None):
    """Greedy-draft mode: accept while x_k equals the target argmax."""
    return _result((_host or _load_host()).greedy_verify(target_logits, draft_tokens, draft_len, workspace, POISON_OUTPUTS))
