"""Re-use of the memory for temporaries (hlu_debug_check_hazards_ring, no GPU):
with a region small enough that its memory is used many times over, a schedule
either orders every conflicting pair of accesses or is refused.  At the
library's own region sizes the meshes that the race check can replay re-use
little or nothing."""
import numpy as np
import pytest

from test_schedule_hazards import FACTOR, SCHULZ_STEP, _trees, lib  # noqa: F401

AT_ONCE, ACCUMULATED, LIBRARY = 0, 1, -1
# region sizes in elements: refused ones, ones a chunk too small for what
# accumulated updates hold, ones with many passes
RINGS = [30000, 40000, 50000, 60000, 80000, 100000, 150000, 300000, 1000000]


def _check(lib, T, cap, tile, which, form, ring):  # noqa: F811
    _, C, B = T
    rep = np.zeros(15, np.int64)
    st = lib.hlu_debug_check_hazards_ring(len(C), C.ctypes.data, len(B), B.ctypes.data, cap, tile, 16, which, form,
                                          ring, rep.ctypes.data)
    return st, rep


# form of the updates: accumulated, or added at once
@pytest.mark.parametrize("n,leaf,tile,cap,general,which,form,early", [
    (5, 8, 16, 32, False, FACTOR, ACCUMULATED, True),
    (6, 16, 32, 32, False, FACTOR, ACCUMULATED, True),
    (6, 16, 64, 64, False, FACTOR, ACCUMULATED, False),
    (6, 16, 64, 64, False, FACTOR, AT_ONCE, False),
    (5, 16, 32, 32, True, FACTOR, ACCUMULATED, False),
    (5, 8, 16, 32, False, FACTOR, AT_ONCE, False),
    (4, 8, 0, 32, False, FACTOR, AT_ONCE, False),
    (4, 8, 16, 32, False, SCHULZ_STEP, ACCUMULATED, False),
    (5, 16, 64, 32, False, SCHULZ_STEP, ACCUMULATED, False),
    (5, 32, 64, 32, True, SCHULZ_STEP, ACCUMULATED, False),
])
def test_reused_memory_is_ordered_or_refused(lib, n, leaf, tile, cap, general, which, form, early):  # noqa: F811
    T = _trees(n, leaf, general)
    runs = []
    for ring in [0] + RINGS:
        st, rep = _check(lib, T, cap, tile, which, form, ring)
        assert st == 0 or (ring > 0 and st == 6), (ring, st, rep)
        if st == 0:
            assert rep[3] == 0 and rep[8] == 0
            runs.append(rep)
    assert runs[0][13] == form
    assert max(r[11] for r in runs if r[13] == form) >= 5
    if early:  # pieces added early keep the memory of accumulated updates free
        assert any(r[12] > 0 and r[13] for r in runs)


def test_bad_arguments(lib):  # noqa: F811
    _, C, B = _trees(3, 16)
    rep = np.zeros(15, np.int64)
    args = (len(C), C.ctypes.data, len(B), B.ctypes.data, 32, 0, 16, FACTOR)
    assert lib.hlu_debug_check_hazards_ring(*args, AT_ONCE, -1, rep.ctypes.data) == 1
    assert lib.hlu_debug_check_hazards_ring(*args, 2, 0, rep.ctypes.data) == 1
    assert lib.hlu_debug_check_hazards_ring(*args, AT_ONCE, 0, None) == 1


@pytest.mark.parametrize("n,leaf", [(4, 16), (4, 8), (5, 16)])
def test_one_truncation_per_step_without_tiles(lib, n, leaf):  # noqa: F811
    """Factored in the block tree's own leaves, a chain of truncations meets each
    diagonal leaf's elimination once: the updates of the steps are not
    truncated one after the other in every target."""
    T = _trees(n, leaf)
    st, rep = _check(lib, T, 32, 0, FACTOR, LIBRARY, 0)
    leaves = int((T[1][:, 8] < 0).sum())
    assert st == 0 and 0 < rep[14] <= leaves, (rep[14], leaves)
