"""Compiles a few kernels of csrc/ behind a C entry of a test's own, for tests
that have to see one kernel's arrays and not a whole call's result."""
import ctypes
import subprocess

from paper_2409_12708_gb300 import build


def compile_kernels(folder, source):
    """source (CUDA, with csrc/ on the include path) as a loaded shared library."""
    cu, so = folder / "kernels.cu", folder / "kernels.so"
    cu.write_text(source)
    cmd = [build.nvcc(), build.ARCH, *build.FLAGS, "-I", build.SRC, "-shared", "-o", str(so), str(cu)]
    done = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if done.returncode != 0:
        raise RuntimeError(done.stdout.decode(errors="replace"))
    return ctypes.CDLL(str(so))


def pointer(tensor):
    return ctypes.c_void_p(tensor.data_ptr())
