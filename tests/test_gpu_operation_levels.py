"""rf_apply refuses, on the host, the operations a level does not have: the
coarsest of several levels is kept as its inverse only, so it has no smoother
sweep and no residual."""
import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_coarsest_level_has_no_smoother_and_no_residual(precision):
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    prob = I.random_problem(3, (9, 9, 9), 91)
    g = rf.Grid(prob)
    g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
    g.gmg_setup([0.1], rf.gmg_opts(2, "gs8", precision=precision))
    v = np.ones(2 * g.nv)
    for op in (rf.RF_OP_SMOOTH, rf.RF_OP_RESIDUAL):
        with pytest.raises(rf.RFError):
            g.apply(op, 1, 0, v, v)
        assert np.isfinite(g.apply(op, 0, 0, v, v)).all()
    g.close()
