"""Shared libraries that GPU tests build from the package's own sources."""
import ctypes
import subprocess

from paper_1804_08923_gb300 import build as b


def shared(src, out, *extra):
    """Compiles src (with the package's flags and include paths) into the shared library out and loads it."""
    cmd = [b.nvcc(), "-shared", "-o", str(out), str(src)] + b.flags() + list(extra)
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    assert r.returncode == 0, r.stdout.decode(errors="replace")
    return ctypes.CDLL(str(out))


def wrapped(src, out, functions):
    """The package's library with src linked between its host code and the functions named {macro: C++ name}:
    src defines WRAP_<macro>, which is called in the function's place, and may call REAL_<macro>."""
    import os
    b.build()
    objs = [os.path.join(b.HERE, "_build", s.replace(".cu", ".o")) for s in b.SOURCES]
    undefined = subprocess.run(["nm", "-u", objs[-1]], stdout=subprocess.PIPE, check=True).stdout.decode().split()
    extra = []
    for macro, name in functions.items():
        sym, = [s for s in undefined if s.startswith(f"_ZN4lbcm{len(name)}{name}E")]
        extra += [f"-DWRAP_{macro}=__wrap_{sym}", f"-DREAL_{macro}=__real_{sym}", "-Xlinker", f"--wrap={sym}"]
    return shared(src, out, *extra, *objs)
