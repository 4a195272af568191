"""Rounding of the device functions that the step kernels share, against what they stand for."""
import ctypes as C
import os

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import native
    L = native.shared(os.path.join(os.path.dirname(__file__), "arithmetic.cu"),
                      tmp_path_factory.mktemp("arithmetic") / "arithmetic.so", "-fmad=false")
    L.reciprocals.argtypes = [C.c_uint, C.c_uint, C.c_void_p]
    L.momentum.argtypes = [C.c_int, C.c_void_p]
    return L


def sums(fn, n, *args):
    import torch
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert fn(*args, out.data_ptr()) == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("exponent", [-20, -1, 0, 3, 40])
def test_reciprocals(lib, exponent):
    """rcp_newton gives 1/x, the nearest float, for every mantissa; rsqrt_newton is on average nearer to
    1/sqrt(x) than a division by the square root, which rounds twice."""
    s = sums(lib.reciprocals, 3, (127 + exponent) << 23, 2 << 23)  # two binades: even and odd exponents
    assert s[0] == 0
    assert s[1] < s[2]


def test_momentum_sums(lib):
    """The momentum of 27 populations summed by classes of c_z, against the sum over opposite pairs.
    x and y are paired within the classes.  For z a class enters as the axis population a, its two
    pairs of faces fx, fy and its four corners k, which are subtracted from the other class's one by
    one.  Squared roundings per class, in units of that of a = f_r + f_b (2/27): a 1, fx and fy (half
    its binade) 1/4 each, the four face populations and the corners 1/16 and less, together below 1.9;
    over opposite pairs a 1 and the populations' 1/16 and less, above 1.25.  So rms is below
    sqrt(1.9 / 1.25) = 1.24 of the pairs'.  Adding a class's faces and corners up first costs another
    1 each: 1.7."""
    s = sums(lib.momentum, 6, 1 << 20)
    for k in range(3):
        assert s[k] <= 1.24 ** 2 * s[3 + k], ("xyz"[k], (s[k] / s[3 + k]) ** 0.5)
