"""The helpers the kernels share with the host (csrc/spdp_hostdev.h), compiled for the host and
run without a GPU: the split of the GTiles over the CTAs at the limits of its 32-bit arithmetic,
and the range check of the checked build on made-up indices (its firing path is only ever
exercised here, never by feeding bad data to a GPU)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    out = tmp_path_factory.mktemp("hostdev") / "libhostdev_shim.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                    "-o", str(out), os.path.join(ROOT, "tests", "hostdev_shim.cpp")], check=True)
    L = ctypes.CDLL(str(out))
    L.shim_range_begin.restype = ctypes.c_uint
    L.shim_range_begin.argtypes = [ctypes.c_uint] * 3
    L.shim_range_owner.argtypes = [ctypes.c_uint] * 3
    L.shim_span_ok.argtypes = [ctypes.c_ulonglong] * 3
    return L


@pytest.mark.parametrize("ngt,P", [(1, 1), (7, 3), (4096, 148), (57344, 148), (11008, 1000), ((1 << 22) - 1, 1024),
                                   ((1 << 22) - 1, 1023), (1 << 21, 1024)])
def test_ranges_partition_the_gtiles_and_owner_inverts_them(H, ngt, P):
    begins = [H.shim_range_begin(ngt, P, c) for c in range(P + 1)]
    assert begins[0] == 0 and begins[-1] == ngt
    assert all(a <= b for a, b in zip(begins, begins[1:]))
    assert begins == [ngt * c // P for c in range(P + 1)]            # no 32-bit wrap at the limits
    probe = sorted({0, ngt - 1, ngt // 2, ngt // 3} | {b for b in begins if b < ngt} | {b - 1 for b in begins if b >= 1})
    for g in probe:
        c = H.shim_range_owner(ngt, P, g)
        assert 0 <= c < P and begins[c] <= g < begins[c + 1], (g, c)


def test_owner_needs_more_than_32_bits_at_the_limits():
    """Why range_owner is 64-bit: its numerator passes 2^32 for the last GTiles at the largest sizes."""
    ngt, P = (1 << 22) - 1, 1024
    assert (ngt * P + ngt - 1) >= 1 << 32 > ngt * P


def test_span_check_fires_only_outside_the_range(H):
    ok = lambda f, c, l: bool(H.shim_span_ok(f, c, l))
    assert ok(0, 0, 0) and ok(0, 16, 16) and ok(15, 1, 16) and ok(16, 0, 16)
    assert not ok(16, 1, 16) and not ok(0, 17, 16) and not ok(17, 0, 16)
    assert not ok((1 << 64) - 1, 2, 1 << 40)                          # first + count would wrap
    assert H.shim_check_code(3) == -1003 and H.shim_check_code(0) == -1000


@pytest.mark.parametrize("R,C,most", [(1, 1, 148), (1, 64, 148), (2, 1024, 148), (4, 64, 148), (16, 256, 148), (43, 256, 148), (112, 512, 148),
                                      (148, 7, 148), (149, 7, 148), (300, 1, 148), (16, 256, 1), (1, 1, 1), (4096, 1023, 148)])
def test_default_ctas_in_range(H, R, C, most):
    H.shim_default_ctas.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    p = H.shim_default_ctas(R, C, most)
    assert 1 <= p <= min(most, R * C)
    if R * C >= 300 * most:
        assert p > 0.9 * most                          # a large layer uses (nearly) every SM


def test_kernels_touch_only_whole_aligned_pinned_buffers(H):
    """Which host buffers the kernels use directly: all bytes inside one page-locked range, elements on their size."""
    f = H.shim_direct_address
    f.argtypes, f.restype = [ctypes.c_ulonglong] * 6, ctypes.c_ulonglong
    start, size, dev = 0x7F0000000000, 4096, 0x700000000000
    at = lambda off, n, align: f(start + off, n, align, start, size, dev + off)
    assert at(0, 4096, 4) == dev and at(8, 100, 4) == dev + 8 and at(2, 10, 2) == dev + 2 and at(4096, 0, 2) == dev + 4096
    assert at(0, 4097, 2) == 0 and at(4000, 98, 2) == 0 and at(4095, 2, 1) == 0          # runs past the range
    assert at(1, 10, 2) == 0 and at(10002, 4, 4) == 0 and at(10, 40, 4) == 0 and at(2, 4, 4) == 0     # off the element's size
    assert f(start - 8, 4, 4, start, size, dev) == 0                                     # before it
    assert f(start, 4, 4, 0, 0, 0) == 0                                                  # pageable
    assert f(start + 8, (1 << 64) - 4, 4, start, size, dev + 8) == 0                     # a length that would wrap
