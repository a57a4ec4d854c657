"""The coarsest operators' dense inverse (k_gauss_jordan: in-place Gauss-Jordan
with partial pivoting over a thread-block cluster) through
rf_dense_inverse_noalloc, at the edges of its row distribution: fewer rows than
CTAs, whole and ragged rows per CTA for each cluster size (4 up to 50 unknowns,
8 up to 143, 16 above), column counts around multiples of the warp.

Elimination with partial pivoting leaves a forward error of at most a modest
multiple of N u kappa(A) relative to the inverse; 16 N u kappa is asked.
"""
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


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 31, 32, 33, 50, 51, 63, 65, 143, 144, 145, 257])
def test_dense_inverse_matches_library(rf, N):
    rng = np.random.default_rng(N)
    A = rng.standard_normal((N, N)) * 10.0 ** rng.uniform(-3, 3, (N, 1))   # rows of very different size
    st, X = _inverse(rf, A)
    assert st == rf.RF_OK
    ref = np.linalg.inv(A)
    bound = 16 * N * 2.0 ** -53 * np.linalg.cond(A) * np.abs(ref).max()
    assert np.abs(X - ref).max() <= bound, (np.abs(X - ref).max(), bound)
    # zero leading pivots and ties: a scaled cyclic permutation inverts exactly
    P = np.roll(np.eye(N) * 2.0, 1, axis=0)
    st, X = _inverse(rf, P)
    assert st == rf.RF_OK and np.array_equal(X, P.T / 4.0)
    # a repeated row: singular
    if N > 1:
        S = A.copy()
        S[:] = np.round(S[:1])
        assert _inverse(rf, S)[0] == rf.RF_ENONFINITE
        Q = P.copy()
        Q[N - 1, 0] = np.inf
        assert _inverse(rf, Q)[0] == rf.RF_ENONFINITE
