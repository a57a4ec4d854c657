"""The columns of a LIMEX step assemble F in parts of their grid's face workspace and
hold none of their own: what a step adds to an assembled and set-up grid is the
extrapolation table and the columns' vectors.  Their residuals, in a ring of fewer
planes and on parallel streams, give the step that sequential columns give, bit for
bit, in grids of one and of many slabs."""
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


def test_columns_hold_their_vectors_only():
    n = (49, 49, 49)
    nv = n[0] * n[1] * n[2]
    prob = I.random_problem(3, n, 81)
    u = torch.tensor(prob["u0"], device="cuda")
    opts = rf.gmg_opts(4, "jacobi", precision="fp64")
    g = rf.Grid(prob)
    g.assemble(u, True)
    g.gmg_setup([0.1, 0.2, 0.3, 0.4], opts)
    torch.cuda.synchronize()
    held = torch.cuda.memory_allocated()
    g.limex_step(u, 10.0, kappa=4, tol=1e9, gmg=opts, rtol=1e-9)
    torch.cuda.synchronize()
    added = torch.cuda.memory_allocated() - held
    # a column: 8 assembly vectors of 8 B, 9 of 16 B, 4 preconditioner vectors and 4 per level (8/7) of 16 B
    column = nv * (8 * 8 + 9 * 16 + 4 * 16 + 4 * 16 * 8 / 7)
    assert added <= 4 * 16 * nv + 3 * (1.1 * column + 1e6), (added, column)
    g.close()


PROBLEMS = {
    "2d-9": (lambda: I.random_problem(2, (9, 9), 82), 2, 5.0),
    "3d-5": (lambda: I.random_problem(3, (5, 5, 5), 82), 2, 5.0),
    "3d-33": (lambda: I.lognormal_box(33, 82), 4, 10.0),
    "3d-97": (lambda: I.lognormal_box(97, 82), 5, 10.0),
    "2d-layers": (lambda: I.case4_analogue((129, 65)), 5, 3600.0),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_concurrent_columns_equal_sequential_ones(name, monkeypatch):
    make, levels, H = PROBLEMS[name]
    prob = make()
    opts = rf.gmg_opts(levels, "gs8", precision="fp32")
    out = []
    for batch, concurrent in (("0", "1"), ("0", "0"), ("1", "0")):
        monkeypatch.setenv("RF_LIMEX_BATCH", batch)
        monkeypatch.setenv("RF_LIMEX_CONCURRENT", concurrent)
        g = rf.Grid(prob)
        u = torch.tensor(prob["u0"], device="cuda")
        for h in (H, 1.2 * H):
            info = g.limex_step(u, h, kappa=4, tol=1e9, gmg=opts, rtol=1e-10)
            assert info["status"] == rf.RF_OK and info["accepted"]
        out.append(u.cpu().numpy())
        g.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
