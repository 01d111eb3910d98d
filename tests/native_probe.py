"""Compiles a few lines of host code against the library's internal headers into a shared object
(nvcc, linked with libgs.so), for tests of rules and launchers that the C ABI does not reach."""
import ctypes
import subprocess

from paper_2604_12942_gb300 import build


def load(tmp_path, source):
    lib = build.build()
    src, so = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text('#include "gs_kernels.cuh"\n' + source)
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I" + build.CSRC, "-shared", "-o", str(so),
                                                                     str(src), lib], check=True)
    return ctypes.CDLL(str(so))
