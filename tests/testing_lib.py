"""Access to the TEST build of the library (csrc/testing.h): the CUDA-core cross-check kernel, the
kernel/split overrides and the wait-timeout probe.  Test infrastructure; the product never loads it."""
from __future__ import annotations

import contextlib
import ctypes

from paper_2505_20776_b200 import api, build

_TLIB = None


def load_testing_lib() -> ctypes.CDLL:
    global _TLIB
    if _TLIB is None:
        L = api.bind(build.build_testing())
        L.specext_test_set_tuning.restype = ctypes.c_int
        L.specext_test_set_tuning.argtypes = [ctypes.c_int32, ctypes.c_int32]
        L.specext_test_wait_timeout.restype = ctypes.c_int
        L.specext_test_wait_timeout.argtypes = [ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p]
        L.specext_test_slow_kernel.restype = ctypes.c_int
        L.specext_test_slow_kernel.argtypes = [ctypes.c_int64, ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p]
        L.specext_test_wait_limit.restype = ctypes.c_int64
        L.specext_test_wait_limit.argtypes = []
        L.specext_test_settle.restype = ctypes.c_int
        L.specext_test_settle.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
        L.specext_test_settle_cycles.restype = ctypes.c_int64
        L.specext_test_settle_cycles.argtypes = []
        L.specext_test_plan.restype = ctypes.c_int
        L.specext_test_plan.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p]
        _TLIB = L
    return _TLIB


def plan(Hq, Hkv, D, T, L, C=32, scored=False, length_on_device=False):
    """(kernel, size of its clusters, rows of Q per CTA, key tiles per worker) of a call on contiguous tensors."""
    d = api.AttnDesc()
    d.n_q_heads, d.n_kv_heads, d.head_dim = Hq, Hkv, D
    d.prefix_len, d.n_tree, d.chunk_size = L, T, C
    d.softmax_scale, d.want_chunk_score = 0.0, int(scored)
    d.q_stride_t, d.kv_stride_l, d.tkv_stride_t, d.o_stride_t = Hq * D, Hkv * D, Hkv * D, Hq * D
    d.q_stride_h = d.kv_stride_h = d.tkv_stride_h = d.o_stride_h = D
    out = (ctypes.c_int32 * 4)()
    assert load_testing_lib().specext_test_plan(ctypes.byref(d), int(length_on_device), out) == 0
    return tuple(out)


@contextlib.contextmanager
def tuned(attn_kernel: int = 0, min_tiles_per_cta: int = 0):
    """Inside the block the binding's calls go to the test library with the given overrides."""
    L = load_testing_lib()
    saved = api._LIB
    assert L.specext_test_set_tuning(attn_kernel, min_tiles_per_cta) == 0
    api._LIB = L
    try:
        yield L
    finally:
        L.specext_test_set_tuning(0, 1)
        api._LIB = saved
