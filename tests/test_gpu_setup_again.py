"""A set-up that follows a new assembly with an unchanged shape takes the
previous hierarchy's buffers, coarse masks and captured iterations again.  Its
solves must equal, bit for bit, those of a grid that is set up for the first
time: with the same and with other shifts, sweeps and states, after a solve
that ended in non-finite values, and for the columns and members of LIMEX
steps.  Options that change the shape build a new hierarchy.
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


def _solve(g, u, shifts, opts, sh):
    F, x = torch.empty_like(u), torch.empty_like(u)
    g.assemble(u, True, F)
    g.gmg_setup(shifts, opts)
    info = g.solve(sh, F, x, rtol=1e-11)
    assert info["status"] == rf.RF_OK, info
    return x.cpu().numpy()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("n,levels", [((17, 13, 9), 2), ((33, 33, 33), 4), ((65, 33, 1), 5)])
def test_repeated_setups_equal_first_ones(n, levels, precision):
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 61)
    u0 = torch.tensor(prob["u0"], device="cuda")
    u1 = u0.clone()
    u1[1::2] *= 0.9
    steps = [(u0, [0.1], "gs8", 2, 0), (u1, [0.1], "gs8", 2, 0), (u1, [0.2], "gs8", 2, 0), (u0, [0.2], "gs8", 1, 0),
             (u0, [0.1, 0.2], "gs8", 2, 1), (u0, [0.1, 0.2], "jacobi", 2, 1), (u1, [0.1, 0.2], "jacobi", 2, 0)]
    g = rf.Grid(prob)
    for k, (u, shifts, smoother, nu, sh) in enumerate(steps):
        opts = rf.gmg_opts(levels, smoother, nu1=nu, precision=precision)
        got = _solve(g, u, shifts, opts, sh)
        fresh = rf.Grid(prob)
        want = _solve(fresh, u, shifts, opts, sh)
        fresh.close()
        assert np.array_equal(got, want), k
        if k == 1:                              # a failed solve leaves NaN in the vectors
            bad = torch.full_like(u, float("nan"))
            bad[2:] = 1.0
            with pytest.raises(rf.RFError):
                g.solve(0, bad, torch.empty_like(u))
            g.apply(rf.RF_OP_VCYCLE, 0, 0, bad.cpu().numpy())
    g.close()


def test_repeated_limex_and_ensemble_steps_equal_first_ones():
    probs = [I.random_problem(3, (17, 17, 17), 71), I.random_problem(3, (17, 17, 17), 72)]
    opts = rf.gmg_opts(3, "gs8", precision="fp32")

    def steps(grids, H):
        us = [torch.tensor(p["u0"], device="cuda") for p in probs]
        st, _ = rf.limex_step_batched(grids, us, H, kappa=3, tol=1e9, gmg=opts, rtol=1e-11)
        assert st == rf.RF_OK
        v = torch.tensor(probs[0]["u0"], device="cuda")
        assert grids[0].limex_step(v, H, kappa=3, tol=1e9, gmg=opts, rtol=1e-11)["status"] == rf.RF_OK
        return [u.cpu().numpy() for u in us + [v]]

    kept = [rf.Grid(p) for p in probs]
    for H in (5.0, 5.0, 7.0):
        got = steps(kept, H)
        fresh = [rf.Grid(p) for p in probs]
        want = steps(fresh, H)
        for g in fresh:
            g.close()
        for a, b in zip(got, want):
            assert np.array_equal(a, b), H
