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
