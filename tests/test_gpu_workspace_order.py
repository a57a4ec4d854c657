"""F alone, assembled on one stream, and a multigrid set-up on another share the grid's
face workspace and nothing else: the set-up waits for the residual, and both results
equal those of calls one after another, bit for bit."""
import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")


@pytest.mark.parametrize("make,levels", [(lambda: I.lognormal_box(97, 91), 5), (lambda: I.lognormal_box(33, 91), 4)])
def test_residual_and_setup_on_two_streams(make, levels):
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    prob = make()
    g = rf.Grid(prob)
    u = torch.tensor(prob["u0"], device="cuda")
    w = u.clone()
    w[1::2] *= 0.8
    b = np.random.default_rng(2).standard_normal(u.numel())
    opts = rf.gmg_opts(levels, "gs8", precision="fp32")
    F, want = torch.empty_like(u), torch.empty_like(u)
    g.assemble(w, False, want)
    g.assemble(u, True)
    g.gmg_setup([0.1], opts)
    cycle = g.apply(rf.RF_OP_VCYCLE, 0, 0, b)
    other = torch.cuda.Stream()
    for _ in range(4):
        g.assemble(u, True)
        torch.cuda.synchronize()
        rf.rf_assemble(g.handle, w.data_ptr(), 0, F.data_ptr(), other.cuda_stream)
        g.gmg_setup([0.1], opts)                # on the grid's stream
        torch.cuda.synchronize()
        assert torch.equal(F, want)
        assert np.array_equal(g.apply(rf.RF_OP_VCYCLE, 0, 0, b), cycle)
    g.close()


def test_residual_can_still_be_captured():
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    prob = I.lognormal_box(17, 92)
    g = rf.Grid(prob)
    u = torch.tensor(prob["u0"], device="cuda")
    F, want = torch.empty_like(u), torch.empty_like(u)
    s = torch.cuda.Stream()
    g.assemble(u, False, want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        rf.rf_assemble(g.handle, u.data_ptr(), 0, F.data_ptr(), s.cuda_stream)
    F.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(F, want)
    g.assemble(u, True)
    g.gmg_setup([0.1], rf.gmg_opts(3, "gs8", precision="fp32"))
    x = torch.empty_like(u)
    assert g.solve(0, F, x, rtol=1e-10)["status"] == rf.RF_OK
    g.close()
