"""The marching level operator refuses a Chebyshev step in place, of the iterate and of the direction: its
16-byte row copies read entries that neighbouring blocks write (host check, nothing is launched)."""
import ctypes as C

import pytest

from paper_1907_06696_gb300 import build as B
from paper_1907_06696_gb300 import capi
from test_outer_host import host_build


@pytest.mark.parametrize("dst_is_src,d_new_is_d", [(1, 0), (0, 1), (1, 1)])
def test_step_in_place_is_refused(tmp_path_factory, dst_is_src, d_new_is_d):
    B.build()
    C.CDLL(capi.LIB_PATH, mode=C.RTLD_GLOBAL)
    assert host_build(tmp_path_factory, "march_host.cpp").march_refuses(dst_is_src, d_new_is_d) == 1
