"""Solves that fail inside the iteration leave non-finite values in the hierarchy's
vectors.  The next set-up takes the same buffers again, and its solves must equal,
bit for bit, those of a new grid: after a single solve, after the columns of a
LIMEX step, and after a batch of which one member failed.
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


def _solve(g, u, opts):
    F, x = torch.empty_like(u), torch.empty_like(u)
    g.assemble(u, True, F)
    g.gmg_setup([0.1], opts)
    assert g.solve(0, F, x, rtol=1e-11)["status"] == rf.RF_OK
    return x.cpu().numpy()


@pytest.mark.parametrize("smoother", ["gs8", "jacobi"])
@pytest.mark.parametrize("precision,size", [("fp32", 1e60), ("fp16", 1e60), ("fp64", 1e152)])
@pytest.mark.parametrize("n,levels", [((17, 13, 9), 2), ((33, 33, 33), 4), ((65, 33, 1), 5)])
def test_setup_after_a_solve_that_overflows(n, levels, precision, size, smoother):
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 63)
    u = torch.tensor(prob["u0"], device="cuda")
    opts = rf.gmg_opts(levels, smoother, precision=precision)
    g = rf.Grid(prob)
    want = _solve(g, u, opts)
    bad = torch.full_like(u, size)                   # finite, |b|^2 too, but no preconditioned iterate is
    with pytest.raises(rf.RFError):
        g.solve(0, bad, torch.empty_like(u), rtol=1e-11)
    assert np.array_equal(_solve(g, u, opts), want)
    g.close()


@pytest.mark.parametrize("batched", [False, True])
def test_setup_after_limex_steps_that_overflow(batched, monkeypatch):
    monkeypatch.setenv("RF_LIMEX_BATCH", "1" if batched else "0")
    probs = [I.random_problem(3, (17, 17, 17), 73), I.random_problem(3, (17, 17, 17), 74)]
    opts = rf.gmg_opts(3, "gs8", precision="fp32")
    kw = dict(kappa=3, tol=1e9, gmg=opts, rtol=1e-11)

    def states(huge):
        us = [torch.tensor(p["u0"], device="cuda") for p in probs]
        if huge:
            us[1][0::2] = 1e60 * (1.0 + torch.arange(us[1].numel() // 2, device="cuda") % 7)
        return us

    def good(grids):
        us = states(False)
        st, _ = rf.limex_step_batched(grids, us, 5.0, **kw)
        assert st == rf.RF_OK
        v = torch.tensor(probs[1]["u0"], device="cuda")
        assert grids[1].limex_step(v, 5.0, **kw)["status"] == rf.RF_OK
        return [u.cpu().numpy() for u in us + [v]]

    grids = [rf.Grid(p) for p in probs]
    want = good(grids)
    us = states(True)
    before = us[1].clone()
    failed = None
    try:
        st, infos = rf.limex_step_batched(grids, us, 5.0, **kw)
        failed = st != rf.RF_OK
    except rf.RFError:
        failed = True
    assert failed and torch.equal(us[1], before)
    with pytest.raises(rf.RFError):
        grids[1].limex_step(us[1], 5.0, **kw)
    for a, b in zip(good(grids), want):
        assert np.array_equal(a, b)
    for g in grids:
        g.close()
