"""Rules of the double-float Gram-Schmidt passes (csrc/gs.cuh), walked through on the host.

GS_LAG writes row j, the last of k rows, while it reads them, so every entry pair of that row must be read by the
group of threads that writes it and by no other, also in the last sweep, where lanes are left over.

The second projection in single precision, with coefficients at the limit up to which it is taken, errs by
less than 2^-53 of the entry's largest |v_i| (bound beside gs_small), whatever the rows hold."""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest

from test_outer_host import host_build


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = host_build(tmp_path_factory, "gs_host.cpp")
    L.gs_shared_pair.restype, L.gs_shared_pair.argtypes = C.c_longlong, [C.c_size_t, C.c_uint] + [C.c_int] * 3
    L.gs_small_limit.restype = C.c_double
    L.gs_small_sum.restype, L.gs_small_sum.argtypes = C.c_double, [C.c_int, C.c_int, C.c_void_p, C.c_void_p]
    return L


@pytest.mark.parametrize("tpe,rb,k", [(1, 4, 1), (1, 4, 4), (1, 16, 14), (2, 12, 17), (2, 12, 24), (2, 16, 25), (4, 10, 33),
                                      (4, 16, 57), (4, 16, 64)])
@pytest.mark.parametrize("blocks", [1, 3, 456])
@pytest.mark.parametrize("n", [1, 2, 33, 255, 1093, 4096, 15738])
def test_the_row_written_is_read_by_its_own_threads_only(lib, n, blocks, tpe, rb, k):
    assert lib.gs_shared_pair(n, blocks, tpe, rb, k) == -1


@pytest.mark.parametrize("tpe,rb", [(1, 4), (1, 16), (2, 16), (4, 10), (4, 16)])
@pytest.mark.parametrize("sign", ["same", "mixed"])
@pytest.mark.parametrize("seed", range(20))
def test_single_precision_projection_at_its_limit(lib, tpe, rb, sign, seed):
    g = np.random.default_rng(1000 * seed + 10 * tpe + rb)
    k, limit = tpe * rb, lib.gs_small_limit()
    c = limit * (1.0 - 2.0 ** -7 * g.uniform(0, 1, k))     # close to the limit, not on FP32 numbers
    v = 1.0 - g.uniform(0, 1, k) * (0.5 if seed % 2 else 1.0)
    if sign == "mixed":
        c, v = c * g.choice([-1.0, 1.0], k), v * g.choice([-1.0, 1.0], k)
    got = lib.gs_small_sum(tpe, rb, np.ascontiguousarray(c).ctypes.data, np.ascontiguousarray(v).ctypes.data)
    want = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(c, v))
    assert abs(Fraction(got) - want) <= Fraction(2) ** -53 * Fraction(float(np.abs(v).max()))
