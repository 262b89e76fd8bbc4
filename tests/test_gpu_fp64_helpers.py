"""sqrt_fp64 and div_fp64 of the FP64 pair sums (csrc/sph_pairmath.cuh), which
start from an FP32 seed, against their error bounds over all exponents.

Square root.  The seed is rsqrtf (at most 2 ulp of FP32, 2^-22) of x cut to 23
bits (2^-24 of its root): y is off by d < 1.25 2^-22.  Goldschmidt's step
leaves 1.5 d^2 < 2^-42 in g and in h, and the correction by the residual, which
is exact to 2^-53 of itself, 2^-83; the last FMA rounds once: 0.5 ulp and less
than 2^-29 ulp.  So the result is the nearest double or, next to a tie, its
neighbour.

Division.  The reciprocal's seed (2 ulp, and x cut to 23 bits) is off by
d < 1.5 2^-22, and y (1 + e + e^2) by d^3 < 2^-64; it is rounded once, by at
most 2^-53 of itself, which is at most 1 ulp of the quotient, and the product
with n once more, by 0.5 ulp: 1.5 ulp and less than 2^-10 ulp.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def helpers(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_03344_gb300 import build
    so = str(tmp_path_factory.mktemp("fp64") / "libfp64_helpers.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-o", so,
                    os.path.join(HERE, "fp64_helpers.cu")], check=True)
    lib = ctypes.CDLL(so)

    def run(x, num):
        t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, num)]
        t += [torch.zeros(len(x), dtype=torch.float64, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        assert lib.helpers(ctypes.c_int64(len(x)), *[ctypes.c_void_p(a.data_ptr()) for a in t]) == 0
        return [a.cpu().numpy() for a in t[2:]]
    return run


def _error_ulp(got, exact):
    """|got - exact| in ulp of got; exact in the widest float numpy has here
    (64 bits of mantissa or more)."""
    return float((np.abs(got.astype(np.longdouble) - exact) / np.spacing(np.abs(got))).max())


def test_errors_over_all_exponents(helpers):
    rng = np.random.default_rng(2)
    e = np.repeat(np.arange(-130, 131), 4000)          # seeds from -120 to 119
    m = rng.uniform(1.0, 2.0, len(e))
    m[::4000] = 1.0                                    # powers of two
    m[1::4000] = np.nextafter(2.0, 1.0)
    x = np.ldexp(m, e)
    num = rng.uniform(-2.0, 2.0, len(e))
    root, quot, ref_root, ref_quot = helpers(x, num)
    xl = x.astype(np.longdouble)
    assert _error_ulp(root, np.sqrt(xl)) < 0.5 + 2.0 ** -9       # 2^-29, and the reference's 2^-11
    assert _error_ulp(quot, num.astype(np.longdouble) / xl) < 1.5 + 2.0 ** -9
    # the library's, correctly rounded, for both bounds' sake
    assert np.abs(root.view(np.int64) - ref_root.view(np.int64)).max() <= 1
    assert np.abs(quot.view(np.int64) - ref_quot.view(np.int64)).max() <= 2


def test_outside_the_seeds_range_the_library(helpers):
    tiny = np.finfo(np.float64).tiny
    b = [2.0 ** -120, 2.0 ** 120]
    x = np.array([0.0, 5e-324, tiny / 2, tiny, 1e-300, 1e300, np.finfo(np.float64).max, np.inf, np.nan,
                  np.nextafter(b[0], 0.0), b[1], np.nextafter(b[1], np.inf), -1.0, -b[0]])
    num = np.full(len(x), 3.0)
    root, quot, ref_root, ref_quot = helpers(x, num)
    assert np.array_equal(root, ref_root, equal_nan=True)
    assert np.array_equal(quot, ref_quot, equal_nan=True)
    # and the last ones inside it
    x = np.array([b[0], np.nextafter(b[0], 1.0), np.nextafter(b[1], 0.0), b[1] / 2])
    root, quot, ref_root, ref_quot = helpers(x, np.full(4, 3.0))
    assert np.abs(root.view(np.int64) - ref_root.view(np.int64)).max() <= 1
    assert np.abs(quot.view(np.int64) - ref_quot.view(np.int64)).max() <= 2
