"""The kernels that a specialised context compiles at its first call need no CUDA
header: their source compiles without an include path (reading the half and
bfloat16 headers cost every variant 12 ms)."""
import ctypes
import os

import pytest

import test_spec_source as source
from paper_1409_5574_gb300 import build


@pytest.mark.parametrize("expr,extra", source.CASES, ids=[str(i) for i in range(len(source.CASES))])
def test_kernel_source_compiles_without_cuda_headers(expr, extra):
    nv = source._nvrtc()
    texts = [open(p, "rb").read() for p in build.SPEC_SOURCES]
    names = [os.path.basename(p).encode() for p in build.SPEC_SOURCES]
    nh = len(texts) - 1
    prog = ctypes.c_void_p()
    assert nv.nvrtcCreateProgram(ctypes.byref(prog), texts[0], names[0], nh,
                                 (ctypes.c_char_p * nh)(*texts[1:]),
                                 (ctypes.c_char_p * nh)(*names[1:])) == 0
    assert nv.nvrtcAddNameExpression(prog, expr) == 0
    opts = [b"-arch=sm_103a", b"-std=c++17", b"-default-device"] + [
        d.encode() for d in source.DEFINES + extra]
    rc = nv.nvrtcCompileProgram(prog, len(opts), (ctypes.c_char_p * len(opts))(*opts))
    n = ctypes.c_size_t()
    nv.nvrtcGetProgramLogSize(prog, ctypes.byref(n))
    log = ctypes.create_string_buffer(n.value + 1)
    nv.nvrtcGetProgramLog(prog, log)
    nv.nvrtcDestroyProgram(ctypes.byref(prog))
    assert rc == 0, log.value.decode(errors="replace")[:2000]
