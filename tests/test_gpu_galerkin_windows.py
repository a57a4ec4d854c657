"""The Galerkin operators (k_galerkin) where its windows differ: one window,
several (a plane kept between them), 2D and 3D, the smallest grids, and a second
coarsening from a full mass stencil.  With FP64 storage the level operator must
act as P^T A P on the unknowns of the correction space, through the transfers
and the finer level's residual: A_c x = P^T A P x for any x that vanishes in
Dirichlet p_w unknowns; the coarse Dirichlet rows are the identity.

Both sides sum the same at most 27 x 27 products per entry in FP64 in different
orders; 1e-12 of the largest value of a component covers a few hundred
roundings of terms that do not cancel below 1/10.
"""
import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("n,levels", [((3, 3, 1), 2), ((3, 3, 3), 2), ((9, 5, 1), 3), ((17, 9, 5), 3), ((33, 9, 17), 3),
                                      ((257, 257, 17), 5), ((8193, 641, 1), 8)])
def test_level_operators_act_as_ptap(n, levels):
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 41)
    g = rf.Grid(prob)
    g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
    shift = 0.1
    g.gmg_setup([shift], rf.gmg_opts(levels, "jacobi", precision="fp64"))
    m, dirv = np.array(n), np.asarray(prob["dir"]).astype(bool).reshape(n[2], n[1], n[0])
    rng = np.random.default_rng(5)
    for level in range(max(1, levels - 2)):
        c = np.where(m > 1, (m - 1) // 2 + 1, 1)
        dc = dirv[::2, ::2, ::2] if dim == 3 else dirv[:, ::2, ::2]
        nf, nc = 2 * int(np.prod(m)), 2 * int(np.prod(c))
        x = rng.standard_normal(nc)
        x[0::2][dc.ravel()] = 0.0
        px = g.apply(rf.RF_OP_PROLONG, level, 0, x, np.zeros(nf), out_len=nf)
        apx = -g.apply(rf.RF_OP_RESIDUAL, level, 0, np.zeros(nf), px, out_len=nf)
        want = g.apply(rf.RF_OP_RESTRICT, level, 0, apx, out_len=nc)
        if level + 1 < levels - 1:
            got = -g.apply(rf.RF_OP_RESIDUAL, level + 1, 0, np.zeros(nc), x, out_len=nc)
        else:                                   # the coarsest level is solved: its inverse undoes P^T A P x
            got, want = x, g.apply(rf.RF_OP_COARSE, level + 1, 0, want, out_len=nc)
        got = got.copy()
        got[0::2][dc.ravel()] = 0.0             # identity rows meet x = 0
        want[0::2][dc.ravel()] = 0.0
        tol = 1e-12 if level + 1 < levels - 1 else 1e-6    # (through the inverse: times its condition)
        for a in range(2):
            assert np.abs(got[a::2] - want[a::2]).max() <= tol * max(np.abs(want[a::2]).max(), 1e-300), (level, a)
        m, dirv = c, dc
    g.close()
