"""The fixed-point arithmetic of the FP64 kernels (csrc/dgpe_fixed.cuh), compiled for the host and
compared with exact integers and with mpmath."""
import ctypes
import os
import subprocess

import pytest

from paper_1610_05329_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_host.so")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                        "-I", os.path.join(build.ROOT, "include"), os.path.join(HERE, "fixed_host.cu"), "-o", so],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def pair(re, im):
    return (ctypes.c_longlong * 2)(re, im)


def hi_lo(h, low):
    return (h << 32) + low


# low words at both ends of a signed word (-2^31 has no 32-bit negative), and around zero
LOW = [-(1 << 31), -(1 << 31) + 1, (1 << 31) - 1, 0, 1, -1]


@pytest.mark.parametrize("dir", [-1, 1])
def test_twiddle_words(lib, dir):
    """a w / 2^64 within the product of the low words (four of at most 2^62, so less than one unit)
    and half a unit of rounding twice: 2 units."""
    out = pair(0, 0)
    for lo_a in LOW:
        for lo_b in LOW:
            for lo_c in LOW:
                for lo_d in LOW:
                    a = (hi_lo(-(1 << 29) + 12345, lo_a), hi_lo((1 << 29) - 99, lo_b))
                    w = (hi_lo((1 << 27) + 7, lo_c), hi_lo(-(1 << 27) + 3, lo_d))
                    lib.host_twiddle(dir, pair(*a), pair(*w), out)
                    wi = w[1] if dir < 0 else -w[1]
                    want = (a[0] * w[0] - a[1] * wi, a[0] * wi + a[1] * w[0])
                    for got, x in zip(out, want):
                        assert abs((got << 64) - x) <= 2 << 64, (a, w)
