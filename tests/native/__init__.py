"""Small shared objects over the library's headers, for tests of parts that the C ABI does not show by themselves."""
import ctypes
import os
import subprocess

from paper_2501_13046_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(name):
    """Compile <name>.cu when it or a header is newer than the object, and load it."""
    src, lib = os.path.join(HERE, name + ".cu"), os.path.join(HERE, "_build", name + ".so")
    if not os.path.exists(lib) or any(os.path.getmtime(f) > os.path.getmtime(lib) for f in [src, *_build.deps()]):
        os.makedirs(os.path.dirname(lib), exist_ok=True)
        tmp = lib + ".tmp%d" % os.getpid()
        subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", src, "-o", tmp], check=True)
        os.replace(tmp, lib)
    return ctypes.CDLL(lib)
