"""Which route a truncation takes and what it may miss (hlu_debug_truncate).

X Y^T has a prescribed spectrum.  Targets up to 128 x 128 are summed densely
(40 columns at most), larger ones sampled: k random samples, at most k - 6
steps, then the stack route."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hlu():
    import __graft_entry__ as g
    g.build()
    from paper_2211_11303_gb300 import hlu as H
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    H.hlu_set_wait_limit_ms(20000)
    return H


def factors(m, n, w, s, seed):
    """X (m x w), Y (n x w), X Y^T = U diag(s) V^T, neither stack orthogonal."""
    rng = np.random.default_rng(seed)
    k = len(s)
    U = np.linalg.qr(rng.standard_normal((m, k)))[0]
    V = np.linalg.qr(rng.standard_normal((n, k)))[0]
    M = np.linalg.qr(rng.standard_normal((w, k)))[0].T * rng.uniform(0.5, 2.0, size=(1, w))
    return (U * s) @ M, (np.linalg.pinv(M) @ V.T).T


def shelf(w, big, height, eps):
    """`big` values down to 5 eps, the rest at height * eps."""
    return np.concatenate([np.logspace(0, np.log10(5 * eps), big), np.full(w - big, height * eps)])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_only_truncations_that_reach_the_stack_are_counted(hlu, prec):
    P = hlu.HLU_FP64 if prec == "fp64" else hlu.HLU_FP32
    eps = 1e-4
    # more values above eps than the dense route keeps, fewer than the samples find
    X, Y = factors(128, 128, 48, shelf(48, 44, 1e-3, eps), 1)
    Xd, _, st = hlu.debug_truncate(X, Y, eps, cap=64, precision=P, piece_cols=48)
    assert Xd.shape[1] == 44 and st[5] == 0
    # as many values above eps as there are samples: neither route can keep them
    X, Y = factors(128, 128, 60, np.logspace(0, np.log10(2 * eps), 60), 2)
    Xd, _, st = hlu.debug_truncate(X, Y, eps, cap=64, precision=P, piece_cols=30)
    assert Xd.shape[1] == 60 and st[5] == 1
