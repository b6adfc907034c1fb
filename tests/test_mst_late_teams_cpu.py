"""Which of a block's teams of the m-sequence transform start late: some, never all."""
import ctypes as C

import pytest


@pytest.mark.parametrize("r, teams, two_rounds, want",
                         [(11, 12, True, 6), (12, 6, True, 3), (13, 3, True, 1), (12, 2, True, 1),
                          (14, 1, True, 1), (12, 1, True, 1),              # no other half
                          (12, 6, False, 6), (10, 6, True, 6)])
def test_late_teams(r, teams, two_rounds, want):
    import paper_2206_05506_gb300 as pk
    f = pk.lib()._ZN4pnce13mst_late_fromEiib
    f.restype, f.argtypes = C.c_int, [C.c_int, C.c_int, C.c_bool]
    assert f(r, teams, two_rounds) == want
