"""Host functions of the library's internal headers, compiled for the CPU tests: the source
text is a translation unit of extern "C" functions that may include csrc/*.cuh."""
import ctypes
import subprocess

from paper_2102_02440_gb300 import build_lib


def compile_probe(tmp_path, source: str) -> ctypes.CDLL:
    cu, so = tmp_path / "probe.cu", tmp_path / "probe.so"
    cu.write_text(source)
    subprocess.check_call([build_lib._nvcc(), *build_lib.ARCH, "-std=c++17", "-Xcompiler", "-fPIC",
                           "--expt-relaxed-constexpr", "-I", build_lib.INCLUDE, "-I", build_lib.CSRC, "-shared",
                           "-o", str(so), str(cu)])
    return ctypes.CDLL(str(so))
