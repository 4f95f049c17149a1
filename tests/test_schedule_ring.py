"""Re-use of the memory for temporaries (hlu_debug_check_hazards_ring, no GPU):
with a region small enough that its memory is used many times over, a schedule
either orders every conflicting pair of accesses or is refused.  At the
library's own region sizes the meshes that the race check can replay re-use
little or nothing."""
import numpy as np
import pytest

from test_schedule_hazards import FACTOR, SCHULZ_STEP, _trees, lib  # noqa: F401

# region sizes in elements: refused ones, ones a chunk too small for what is
# held, ones with many passes
RINGS = [30000, 40000, 50000, 60000, 80000, 100000, 150000, 300000, 1000000]


@pytest.mark.parametrize("n,leaf,tile,cap,general,which", [
    (5, 8, 16, 32, False, FACTOR),
    (6, 16, 32, 32, False, FACTOR),
    (6, 16, 64, 64, False, FACTOR),
    (5, 16, 32, 32, True, FACTOR),
    (4, 8, 0, 32, False, FACTOR),
    (4, 8, 16, 32, False, SCHULZ_STEP),
    (5, 16, 64, 32, False, SCHULZ_STEP),
    (5, 32, 64, 32, True, SCHULZ_STEP),
])
def test_reused_memory_is_ordered_or_refused(lib, n, leaf, tile, cap, general, which):  # noqa: F811
    _, C, B = _trees(n, leaf, general)
    passes = []
    for ring in [0] + RINGS:
        rep = np.zeros(12, np.int64)
        st = lib.hlu_debug_check_hazards_ring(len(C), C.ctypes.data, len(B), B.ctypes.data, cap, tile, 16, which,
                                              ring, rep.ctypes.data)
        assert st == 0 or (ring > 0 and st == 6), (ring, st, rep)
        if st == 0:
            assert rep[3] == 0 and rep[8] == 0
            passes.append(int(rep[11]))
    assert max(passes) >= 5, passes


def test_bad_arguments(lib):  # noqa: F811
    _, C, B = _trees(3, 16)
    rep = np.zeros(12, np.int64)
    args = (len(C), C.ctypes.data, len(B), B.ctypes.data, 32, 0, 16, FACTOR)
    assert lib.hlu_debug_check_hazards_ring(*args, -1, rep.ctypes.data) == 1
    assert lib.hlu_debug_check_hazards_ring(*args, 0, None) == 1
