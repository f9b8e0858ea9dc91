"""What the allocation-free electrostatic solve reports for each way a persistent
solve can end (no GPU needed: the state it reads back is made up here)."""
import ctypes as C

import pytest

from paper_2102_06248_gb300 import fempic as F

NO_CONVERGENCE, BARRIER = 2, 32     # status bits of csrc/internal.h


@pytest.mark.parametrize("done,failed,status,code,text", [
    (1, 0, 0, 0, None),
    (1, 1, NO_CONVERGENCE, 6, "tolerance"),
    (0, 0, 0, 6, "tolerance"),                       # the solve wrote nothing
    (1, 1, BARRIER, 8, "grid barrier"),              # a wait ran out: not a matter of the tolerance
    (0, 0, BARRIER, 8, "grid barrier"),
    (1, 1, BARRIER | NO_CONVERGENCE, 8, "grid barrier"),
])
def test_outcome(done, failed, status, code, text):
    lib = F.load()
    outcome = lib._ZN2fp15noalloc_outcomeEiij        # fp::noalloc_outcome(int, int, uint32_t)
    outcome.argtypes, outcome.restype = [C.c_int, C.c_int, C.c_uint32], C.c_int
    assert outcome(done, failed, status) == code
    if text:
        assert text in lib.pic_last_error().decode()
