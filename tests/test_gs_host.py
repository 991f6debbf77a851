"""Rules of the double-float Gram-Schmidt passes (csrc/gs.cuh), walked through on the host.

GS_LAG writes row j of the basis while it reads it, so every entry pair must be read by the group of
threads that writes it and by no other, also in the last sweep, where lanes are left over."""
import ctypes as C

import pytest

from test_outer_host import host_build


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = host_build(tmp_path_factory, "gs_host.cpp")
    L.gs_shared_pair.restype, L.gs_shared_pair.argtypes = C.c_longlong, [C.c_size_t, C.c_uint, C.c_int]
    return L


@pytest.mark.parametrize("tpe", [1, 2, 4])
@pytest.mark.parametrize("blocks", [1, 3, 456])
@pytest.mark.parametrize("n", [1, 2, 33, 255, 1093, 4096, 15738])
def test_every_pair_is_read_by_its_own_threads_only(lib, n, blocks, tpe):
    assert lib.gs_shared_pair(n, blocks, tpe) == -1
