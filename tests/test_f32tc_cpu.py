"""The FP32 tensor-core kernels compile for sm_103a (no GPU)."""
import ctypes

import pytest

from paper_0911_3456_gb300 import _capi as C


@pytest.mark.parametrize("shape,spec,ok", [
    (((64, 64, 4), (16, 3, 3, 4)), "f32tc", True),
    (((40, 50, 33), (7, 13, 13, 33)), "f32tc", True),
    (((128, 128, 8), (16, 9, 9, 8)), "f32tc:nt=64,r=4,gc=8,jt=9,ru=2", True),
    (((128, 128, 8), (16, 9, 9, 8)), "f32tc:nt=64,r=4,gc=8,jt=9", False),
])
def test_rtcg_check(shape, spec, ok):
    log = ctypes.create_string_buffer(8192)
    st = C.load().fbcorr_rtcg_check(C.I64_3(*shape[0]), C.I64_4(*shape[1]), C.epilogue((0.0, 1.0)), spec.encode(), log,
                                    len(log))
    assert (st == 0) == ok, log.value.decode()
