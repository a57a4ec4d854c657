"""The coarsest operators' inverse (k_lu_cluster and k_lu_inverse_cols) is, to the
last bit, that of LU factors with partial pivoting and substitutions whose sums are
32 lanes' partial sums, as the kernels of one CTA compute it (k_lu, with
RF_LU_CLUSTER=0): against exact emulation of every rounded operation at the sizes
that takes seconds for, and against k_lu beyond, at the edges of the row
distribution and with ties among the pivots.  The elimination of a cluster may not
cost accuracy: its sums are no longer than those of one CTA.
"""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rf():
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2506_04763_gb300 as R
    return R


def _inverse(rf, A):
    d = torch.tensor(A, device="cuda")
    out = torch.full_like(d, float("nan"))
    st = rf.lib().rf_dense_inverse_noalloc(len(A), d.data_ptr(), out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return st, out.cpu().numpy()


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _lane_dot(row, x, c0, c1):
    s = [0.0] * 32
    for c in range(c0, c1):
        s[(c - c0) % 32] = _fma(row[c], x[c], s[(c - c0) % 32])
    for o in (16, 8, 4, 2, 1):
        s = [s[i] + s[i ^ o] for i in range(32)]
    return s[0]


def _emulated_inverse(A):
    N = len(A)
    D = [[float(v) for v in r] for r in A]
    at = list(range(N))
    for c in range(N):
        p = max(range(c, N), key=lambda r: (abs(D[r][c]), -r))
        D[c], D[p] = D[p], D[c]
        at[c], at[p] = at[p], at[c]
        for r in range(c + 1, N):
            m = D[r][c] / D[c][c]
            D[r][c] = m
            for t in range(c + 1, N):
                D[r][t] = _fma(-m, D[c][t], D[r][t])
    X = np.empty((N, N))
    for col in range(N):
        x = [1.0 if at[r] == col else 0.0 for r in range(N)]
        for r in range(1, N):
            x[r] -= _lane_dot(D[r], x, 0, r)
        for r in range(N - 1, -1, -1):
            x[r] = (x[r] - _lane_dot(D[r], x, r + 1, N)) / D[r][r]
        X[:, col] = x
    return X


def _matrix(N, kind):
    rng = np.random.default_rng([N, len(kind)])
    if kind == "scaled":                       # rows of very different size, as p_w and S_n rows are
        return rng.standard_normal((N, N)) * 10.0 ** rng.uniform(-6, 6, (N, 1))
    if kind == "ties":                         # few distinct values: most pivots are chosen among equals
        return rng.integers(-1, 2, (N, N)) + 4.0 * np.roll(np.eye(N), 3, axis=0)
    A = -rng.random((N, N)) * (rng.random((N, N)) < 0.3)       # diagonally dominant, negative off the diagonal
    return A + np.diag(1e-3 - A.sum(1) + np.diag(A))


@pytest.mark.parametrize("kind", ["scaled", "ties", "dominant"])
@pytest.mark.parametrize("N", [1, 2, 5, 16, 33, 51])
def test_inverse_is_lu_and_substitution_to_the_last_bit(rf, N, kind):
    A = _matrix(N, kind)
    st, X = _inverse(rf, A)
    assert st == rf.RF_OK
    assert np.array_equal(X, _emulated_inverse(A))


@pytest.mark.parametrize("kind", ["scaled", "ties", "dominant"])
@pytest.mark.parametrize("N", [3, 4, 31, 32, 50, 52, 64, 143, 144, 145, 250, 257, 289, 511, 512])
def test_cluster_and_one_cta_agree_to_the_last_bit(rf, N, kind, monkeypatch):
    A = _matrix(N, kind)
    a = _inverse(rf, A)
    monkeypatch.setenv("RF_LU_CLUSTER", "0")
    b = _inverse(rf, A)
    assert a[0] == b[0] == rf.RF_OK
    assert np.array_equal(a[1], b[1])
    ref = np.linalg.inv(A)
    bound = 16 * N * 2.0 ** -53 * np.linalg.cond(A) * np.abs(ref).max()
    assert np.abs(b[1] - ref).max() <= bound


def test_a_large_coarsest_level_takes_the_factors_of_one_cta(rf):
    """19 x 19 vertices, 722 unknowns: beyond a cluster's shared memory."""
    from paper_2506_04763_gb300 import inputs as I
    from tests import _helpers as H
    prob = I.random_problem(2, (37, 37), 17)
    g = rf.Grid(prob)
    g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
    g.gmg_setup([0.1, 0.4], rf.gmg_opts(2, "gs8", precision="fp64"))
    rng = np.random.default_rng(4)
    for j in (0, 1):
        A, n = g.export_level(1, j)
        D = H.stencil_to_dense(2, n, np.asarray(A).reshape(19 * 19, 9, 4))
        b = rng.standard_normal(len(D))
        x = g.apply(rf.RF_OP_COARSE, 1, j, b, out_len=len(b))
        inv = np.linalg.inv(D)
        bound = 16 * len(D) * 2.0 ** -53 * np.linalg.cond(D) * np.abs(inv).max() * np.abs(b).sum()
        assert np.abs(x - inv @ b).max() <= bound
    g.close()
