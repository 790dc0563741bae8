"""A CTA of the step kernel whose waits gave up is left by all its consumer
warps at the same barrier: the decision comes out of the barrier, so a flag
raised between two warps' reads of it cannot part them (a warp that stayed
would wait for the others without a limit)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas,rounds", [(1, 1), (152, 200000), (4000, 200000)])
def test_consumer_warps_leave_together(ctas, rounds):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_06908_gb300 import _lib
    lib = _lib.load()
    spread, early = ctypes.c_int(-1), ctypes.c_int(-1)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.fdtd_selftest_leave(ctas, rounds, ctypes.byref(spread), ctypes.byref(early), stream) == 0
    assert spread.value == 0
    if rounds > 1:
        assert early.value > 0


def test_bad_arguments():
    from paper_2207_06908_gb300 import _lib
    lib = _lib.load()
    a, b = ctypes.c_int(), ctypes.c_int()
    for ctas, rounds, p in ((0, 1, a), (65536, 1, a), (1, 0, a), (1, 1000001, a), (1, 1, None)):
        assert lib.fdtd_selftest_leave(ctas, rounds, ctypes.byref(p) if p is not None else None, ctypes.byref(b),
                                       None) == -1
