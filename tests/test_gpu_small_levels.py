"""The kernels of small levels (rows loaded whole, two lanes per row pair in FP64,
colour pairs spread line by line) and the cluster tail with its vectors in
shared memory, at shapes where they can go wrong: lines shorter and longer than
a warp or a block, one or two lines, odd and even counts per parity, fewer lines
than CTAs, levels just below and above the limits of the rules.  Every form
performs the same operations per vertex in the same order, so a V-cycle equals,
bit for bit, the V-cycle of the plain forms: one launch per phase (RF_TAIL_NV=0)
and per colour (RF_GS_PAIRS=0).
"""
import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")

SHAPES = [((3, 3, 1), 2), ((9, 17, 1), 3), ((5, 65, 1), 3), ((577, 5, 1), 3), ((129, 65, 1), 5), ((257, 129, 1), 6),
          ((5, 5, 5), 2), ((9, 5, 17), 3), ((33, 17, 9), 4), ((17, 33, 33), 4), ((65, 33, 33), 4), ((321, 5, 9), 3),
          ((37, 33, 33), 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("smoother,nu", [("gs8", (2, 2)), ("jacobi", (2, 2)), ("jacobi", (1, 2)), ("gs8", (1, 0))])
@pytest.mark.parametrize("n,levels", SHAPES)
def test_small_level_forms_are_bitwise_equal(n, levels, smoother, nu, precision, monkeypatch):
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 51)
    rng = np.random.default_rng(6)
    b = rng.standard_normal(2 * n[0] * n[1] * n[2])
    out = []
    for plain in (False, True):
        if plain:
            monkeypatch.setenv("RF_TAIL_NV", "0")
            monkeypatch.setenv("RF_GS_PAIRS", "0")
        g = rf.Grid(prob)
        g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
        g.gmg_setup([0.1, 0.3], rf.gmg_opts(levels, smoother, nu1=nu[0], nu2=nu[1], precision=precision))
        out.append([g.apply(rf.RF_OP_VCYCLE, 0, j, b) for j in (0, 1)])
        g.close()
    for j in (0, 1):
        assert np.all(np.isfinite(out[0][j]))
        assert np.array_equal(out[0][j], out[1][j]), np.abs(out[0][j] - out[1][j]).max()
