"""Sizes of the workspaces that the queries ask for (no GPU needed): a large
product needs no more scratch than its digits take.

Bound: ceil(8 s / 7) BF16 digits of both operands (the sign-magnitude digits of 7
bits whose products are folded into C on the fly), or 4 GiB where that is more,
and for a block of at most 1024 x 256 entries of C.
"""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1911_11906_gb300 import build
    L = ctypes.CDLL(build.build())
    L.fraclap_dgemm_ozaki_workspace_bytes.restype = ctypes.c_size_t
    L.fraclap_dgemm_ozaki_workspace_bytes.argtypes = [ctypes.c_int64] * 3 + [ctypes.c_int]
    return L


@pytest.mark.parametrize("m,n,k", [(31996, 31996, 31996), (70706, 70706, 70706), (31996, 65535, 31996), (45000, 300, 45000),
                                   (180000, 180000, 64), (2000000, 1, 4000), (16, 16, 200000000), (250, 65535, 250)])
@pytest.mark.parametrize("slices", [1, 5, 6, 7, 8])
def test_slice_products(lib, m, n, k, slices):
    kp = -(-k // 64) * 64
    digits = -(-8 * slices // 7) * 2 * (m + n) * kp
    block = 45 * 4 * 1024 * 256 + 18 * 256 * min(kp, 130048) + 64 * (m + n)
    assert lib.fraclap_dgemm_ozaki_workspace_bytes(m, n, k, slices) <= max(4 << 30, digits + block) + 4096


@pytest.mark.parametrize("slices", [1, 5, 6, 7, 8])
@pytest.mark.parametrize("m,n,k", [(18225, 4096, 18225), (33333, 7, 40001), (40001, 40003, 33), (1, 1, 1)])
def test_a_workspace_of_the_size_asked_for_is_accepted(lib, m, n, k, slices):
    """(sizes are compared in units of 256 bytes)"""
    assert lib.fraclap_dgemm_ozaki_workspace_bytes(m, n, k, slices) % 256 == 0
