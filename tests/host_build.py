"""The host-evaluable rules of csrc/*.h, compiled by the host compiler and called through ctypes."""
import ctypes
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_23733_gb300", "csrc")


def host_lib(tmp_path, source, flags=("-O2",)):
    """A shared library of the C++17 text ``source`` (csrc on the include path)."""
    src, lib = os.path.join(tmp_path, "rules.cpp"), os.path.join(tmp_path, "rules.so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", *flags, "-I", CSRC, src, "-o", lib],
                   check=True)
    return ctypes.CDLL(lib)
