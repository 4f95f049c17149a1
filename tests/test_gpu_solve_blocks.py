"""The triangular solve's kernel and the inverted diagonal blocks it multiplies
with: every right-hand-side count it groups differently, block and tile
remainders, and its bounded wait."""
import numpy as np
import pytest

import synth
from oracle import fem, mesh

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


# N = 26 (one ragged tile), 316 (one block), 665 and 1206 (several blocks with
# low-rank updates between them); leaf sizes that leave 3-row to 64-row units
@pytest.mark.parametrize("n,leaf", [(2, 8), (4, 3), (5, 16), (6, 32), (6, 64)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_columns_do_not_depend_on_their_number(hlu, n, leaf, prec):
    kappa = 3.0
    A = fem.assemble(mesh.interior_edges(n), kappa).toarray()
    N = A.shape[0]
    B = np.stack([synth.normal(300 + j, N) for j in range(17)], axis=1)
    X = np.linalg.solve(A, B)
    h = hlu.hlu_build(n, kappa, leaf, 2.0, 1e-12)
    try:
        hlu.hlu_factor(h, hlu.HLU_FP64 if prec == "fp64" else hlu.HLU_FP32)
        got = {}
        for k in (1, 3, 4, 5, 8, 9, 16, 17):
            b = hlu.colmajor(N, k)
            b.copy_(torch.from_numpy(B[:, :k]))
            x = hlu.colmajor(N, k)
            hlu.hlu_solve(h, b, x)
            got[k] = x.cpu().numpy()
        for k, x in got.items():
            assert np.array_equal(x, got[17][:, :k]), k
        # as the parity tests of a factor at eps -> 0: rounding times the condition
        u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
        bar = max(1e-9, 4 * np.sqrt(N) * np.linalg.cond(A) * u)
        err = np.linalg.norm(got[17] - X, axis=0) / np.linalg.norm(X, axis=0)
        assert err.max() <= bar, (err.max(), bar)
    finally:
        hlu.hlu_destroy(h)


def test_bounded_wait_of_the_solve_reports_a_timeout(hlu):
    st = np.zeros(2, np.int32)
    assert hlu.lib().hlu_debug_solve_wait_timeout(200.0, st.ctypes.data) == 5
    assert st[0] == 5 and st[1] == 0
    h = hlu.hlu_build(3, 2.0, 16, 2.0, 1e-6)  # the device stays usable
    try:
        hlu.hlu_factor(h, hlu.HLU_FP32)
        N = hlu.hlu_n(h)
        b = torch.ones(N, dtype=torch.float64, device="cuda")
        x = torch.empty_like(b)
        assert hlu.gmres_solve(h, b, x, tol=1e-10)["converged"] == 1
    finally:
        hlu.hlu_destroy(h)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_first_solve_of_a_factor_under_capture(hlu, prec):
    """hlu_solve captured in a graph before any other solve of the factor: what
    the solve reads beside the factor belongs to the factorisation, so eager
    solves and replays before and after another factorisation agree."""
    P = hlu.HLU_FP64 if prec == "fp64" else hlu.HLU_FP32
    other = hlu.hlu_build(4, 2.0, 16, 2.0, 1e-4)
    h = hlu.hlu_build(6, 3.0, 16, 2.0, 1e-4)
    try:
        N = hlu.hlu_n(h)
        b = hlu.colmajor(N, 3)
        b.copy_(torch.from_numpy(np.stack([synth.normal(70 + j, N) for j in range(3)], axis=1)))
        x, y = hlu.colmajor(N, 3), hlu.colmajor(N, 3)
        hlu.hlu_factor(other, P)  # loads the solve's kernels
        no = hlu.hlu_n(other)
        hlu.hlu_solve(other, torch.ones(no, dtype=torch.float64, device="cuda"),
                      torch.empty(no, dtype=torch.float64, device="cuda"))
        hlu.hlu_factor(h, P)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            hlu.hlu_solve(h, b, x)
        hlu.hlu_solve(h, b, y)  # eager, before the first replay
        r = torch.empty_like(y)
        hlu.hlu_spmv(h, y, r)
        assert (torch.linalg.norm(r - b) / torch.linalg.norm(b)).item() < 0.1
        for again in (False, True):
            if again:
                hlu.hlu_factor(h, P)
            x.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(x, y)
    finally:
        hlu.hlu_destroy(h)
        hlu.hlu_destroy(other)


def test_solve_bytes_count_what_a_solve_reads(hlu):
    """One solve block (N <= 512): both triangles of its inverse and nothing of
    the factor; more blocks: also the off-diagonal factor, less than the sum of
    all panels and all live words."""
    h = hlu.hlu_build(4, 2.0, 16, 2.0, 1e-4)
    try:
        assert hlu.hlu_solve_bytes(h) == -1
        N = hlu.hlu_n(h)
        assert N <= 512
        for prec, es in ((hlu.HLU_FP32, 4), (hlu.HLU_FP64, 8)):
            hlu.hlu_factor(h, prec)
            # two triangles of units of at most 64 rows: N (N + rows of the unit) words
            assert N * (N + 1) * es <= hlu.hlu_solve_bytes(h) <= N * (N + 64) * es
    finally:
        hlu.hlu_destroy(h)
    h = hlu.hlu_build(8, 2.0, 16, 2.0, 1e-4)
    try:
        hlu.hlu_factor(h, hlu.HLU_FP32)
        N = hlu.hlu_n(h)
        live = hlu.hlu_factor_stats(h)["factor_live_bytes"]
        panels = N * (512 + 64) * 4
        assert N * 64 * 4 < hlu.hlu_solve_bytes(h) < live + panels
    finally:
        hlu.hlu_destroy(h)
