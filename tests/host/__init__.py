"""Host programs that tests compile against the library's internal headers."""
import ctypes
import os
import subprocess

from paper_1707_00516_gb300 import build as Bd

HERE = os.path.dirname(os.path.abspath(__file__))


def compile_against_library(source: str, out: str, *flags: str) -> str:
    """Compile tests/host/<source> and link it with libfastid.so."""
    subprocess.run([Bd._nvcc(), "-std=c++17", "-I", Bd.INCLUDE, "-I", Bd.CSRC, *flags, "-o", out,
                    os.path.join(HERE, source), Bd.build(), "-Xlinker", f"-rpath={Bd.PKG}"], check=True,
                   capture_output=True)
    return out


def ctx_hooks(tmp) -> ctypes.CDLL:
    """tests/host/ctx_hooks.cu as a loaded library."""
    lib = ctypes.CDLL(compile_against_library("ctx_hooks.cu", os.path.join(str(tmp), "ctx_hooks.so"), "-shared",
                                              "-Xcompiler", "-fPIC"))
    lib.hook_fp4_block_bytes.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    lib.hook_fp4_block_bytes.restype = None
    lib.hook_few_rule.argtypes = [ctypes.c_void_p, ctypes.c_int32]
    lib.hook_few_rule.restype = None
    lib.hook_few_stages.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int32]
    lib.hook_few_pays.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int64, ctypes.c_int64]
    lib.hook_plain_fills.argtypes = [ctypes.c_int32, ctypes.c_int32, ctypes.c_int64, ctypes.c_int64]
    lib.hook_kbytes4.argtypes = [ctypes.c_int32]
    return lib
