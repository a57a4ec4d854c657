"""The kernels of small levels against the plain ones (RF_SMALL_NV=0) on the same
levels, each launched on its own (RF_TAIL_NV=0): every sweep and residual of every
level, and whole V-cycles, are equal bit for bit.  Shapes where the small forms can
go wrong: lines shorter and longer than a warp or a block's rounds, odd and even
counts per parity, one line of a parity, fewer lines than SMs and more, a level just
below the limit.  That the two arms run different kernels is seen from the launches
of an FP64 sweep: one per pair of colours on a small level, one per colour else.
"""
import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")

SHAPES = [((3, 3, 1), 2), ((9, 17, 1), 3), ((5, 65, 1), 3), ((577, 5, 1), 3), ((257, 129, 1), 5), ((5, 5, 5), 2),
          ((9, 5, 17), 3), ((33, 17, 9), 4), ((321, 5, 9), 3), ((37, 33, 29), 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("smoother", ["gs8", "jacobi"])
@pytest.mark.parametrize("n,levels", SHAPES)
def test_small_forms_equal_the_plain_kernels_per_level(n, levels, smoother, precision, monkeypatch):
    monkeypatch.setenv("RF_TAIL_NV", "0")
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 53)
    out, sweeps = [], []
    for small in (True, False):
        if not small:
            monkeypatch.setenv("RF_SMALL_NV", "0")
        g = rf.Grid(prob)
        g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
        g.gmg_setup([0.1, 0.3], rf.gmg_opts(levels, smoother, precision=precision))
        rng = np.random.default_rng(8)
        m, res = list(n), []
        for lev in range(levels - 1):
            b, x = rng.standard_normal((2, 2 * int(np.prod(m))))
            for j in (0, 1):
                before = rf.rf_launch_count()
                res.append(g.apply(rf.RF_OP_SMOOTH, lev, j, b, x, out_len=len(b)))
                sweeps.append(rf.rf_launch_count() - before)
                res.append(g.apply(rf.RF_OP_RESIDUAL, lev, j, b, x, out_len=len(b)))
            if lev == 0:
                res += [g.apply(rf.RF_OP_VCYCLE, 0, j, b) for j in (0, 1)]
            m = [(t - 1) // 2 + 1 for t in m]
        out.append(res)
        g.close()
    for k, (a, b) in enumerate(zip(*out)):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b), (k, np.abs(a - b).max())
    if precision == "fp64" and smoother == "gs8":
        half = len(sweeps) // 2
        assert all(a < b for a, b in zip(sweeps[:half], sweeps[half:])), sweeps
