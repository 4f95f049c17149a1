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


def test_fp32_samples_are_not_taken_below_1e6(hlu):
    """Below eps 1e-6 the samples' rounding is too near eps: a spectrum that they
    would give up goes to the stack at once."""
    for eps, redone in ((7e-7, 0), (2e-6, 1)):
        X, Y = factors(200, 180, 60, np.logspace(0, np.log10(2 * eps), 60), 3)
        _, _, st = hlu.debug_truncate(X, Y, eps, cap=64, precision=hlu.HLU_FP32, piece_cols=30)
        assert st[5] == redone, eps


def signs(rows, cols):
    """The samples' coefficients: the hash of the index row * 96 + column."""
    h = (np.arange(rows, dtype=np.int64)[:, None] * 96 + np.arange(cols)).astype(np.uint32)
    h = h + np.uint32(0x9E3779B9)
    for shift, mul in ((16, 0x85EBCA6B), (13, 0xC2B2AE35), (16, 1)):
        h ^= h >> np.uint32(shift)
        h *= np.uint32(mul)
    return np.where(h & np.uint32(1), 1.0, -1.0)


def sampled_steps(A, k, eps, noise=9e-14):
    """(steps, most steps, square of what they miss over (0.1 eps s_1)^2, ratio of
    the last nine pivots) of the sampled route in 64 bits; noise: its FP32
    rounding floor."""
    S = A @ signs(A.shape[1], k)
    left, kend, piv = list(range(k)), min(k - 6, 64, *A.shape), []
    while True:
        n2 = (S[:, left] ** 2).sum(0)
        first = n2.max() if not piv else first
        missed = n2.sum() * k / (first * (k - len(piv)))
        if len(piv) >= kend or missed <= max(0.01 * eps * eps, noise):
            return len(piv), kend, missed / (0.01 * eps * eps), piv[-9] / piv[-1]
        c = left[int(n2.argmax())]
        q = S[:, c] / np.sqrt(n2.max())
        piv.append(np.sqrt(n2.max()))
        left.remove(c)
        S[:, left] -= np.outer(q, q @ S[:, left])


# FP32 ends of the sampled route above its own floor: the last step with up to
# 0.55 eps missed, with up to eps missed when the last pivots are level, and the
# rounding floor of the samples
ENDS = [
    ("last", 200, 180, 64, 22, 0.05, 1e-4),
    ("last", 700, 600, 64, 22, 0.05, 1e-4),
    ("flat", 300, 260, 64, 12, 0.11, 1e-4),
    ("flat", 700, 600, 64, 10, 0.10, 1e-4),
    ("floor", 300, 280, 60, 24, 0.02, 1e-6),
    ("floor", 500, 520, 48, 24, 0.02, 1e-6),
]


@pytest.mark.parametrize("end,m,n,w,big,height,eps", ENDS)
def test_sampled_route_keeps_the_bound_at_each_end(hlu, end, m, n, w, big, height, eps):
    s = shelf(w, big, height, eps)
    X, Y = factors(m, n, w, s, 1)
    F = X @ Y.T
    steps, most, miss, level = sampled_steps(F, 64, eps)
    if end == "last":
        assert steps == most and 2 < miss < 20
    elif end == "flat":
        assert steps == most and 32 < miss < 90 and level < 1.9
    else:
        assert steps + 5 < sampled_steps(F, 64, eps, 0.0)[0]
    Xd, Yd, st = hlu.debug_truncate(X, Y, eps, cap=64, precision=hlu.HLU_FP32, piece_cols=w // 2)
    assert st[0] == 0 and st[5] == 0  # finished by the samples
    assert Xd.shape[1] == big
    # the bound of every truncation: eps, and FP32 rounding of the factors
    rnd = 3e-6 * np.linalg.norm(X, 2) * np.linalg.norm(Y, 2) / s[0]
    assert np.linalg.norm(F - Xd @ Yd.T, 2) <= (1.05 * eps + rnd) * s[0]
