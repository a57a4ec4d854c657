"""The two-pass assembly (faces, then rows) against the one-thread-per-vertex
kernel (RF_ASM_VERTEX=1), which evaluates the same face arithmetic from each
vertex: F, J and M over the shapes where its slabs and edges differ — one cell
per axis, odd and even line lengths, 2D, several slabs along z, slabs along y
(wide, shallow boxes), per-medium laws and the discretisation variants.

Both kernels take the same decisions and round every face derivative alike;
the entries are sums of at most 24 of them in another order, so rows agree
to a few hundred roundings of their largest term (1e-13 of the row's largest
entry covers it, as the terms of these states do not cancel by more than 10x).
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


def _problem(n, seed, scheme=0, laws=False):
    dim = 3 if n[2] > 1 else 2
    p = I.random_problem(dim, n if dim == 3 else n[:2], seed, stress=min(n[:dim]) < 40)
    p["scheme"] = scheme
    return I.mixed_kr_laws(p, seed) if laws else p


@pytest.mark.parametrize("n,scheme,laws", [
    ((2, 2, 1), 0, False), ((3, 2, 1), 0, False), ((34, 19, 1), 0, True), ((801, 5, 1), 2, False),
    ((2, 2, 2), 0, False), ((2, 3, 7), 1, False), ((8, 2, 5), 3, True), ((33, 18, 11), 0, True),
    ((65, 7, 34), 2, False), ((130, 129, 83), 0, False), ((601, 600, 3), 0, False),
])
def test_faces_and_vertex_assembly_agree(n, scheme, laws, monkeypatch):
    prob = _problem(n, 31, scheme, laws)
    u = torch.tensor(prob["u0"], device="cuda")
    out = []
    for mode in ("0", "1"):
        monkeypatch.setenv("RF_ASM_VERTEX", mode)
        g = rf.Grid(prob)
        F, F2 = torch.empty_like(u), torch.empty_like(u)
        g.assemble(u, True, F)
        J, md = g.export_jacobian()
        g.assemble(u, False, F2)
        torch.cuda.synchronize()
        assert torch.equal(F, F2), "F with and without J"
        out.append((F.cpu().numpy(), J, md))
        g.close()
    (F0, J0, m0), (F1, J1, m1) = out
    for a in range(2):
        rows = np.abs(J1[:, :, 2 * a:2 * a + 2]).max(axis=(1, 2)) + 1e-300
        err = np.abs(J0[:, :, 2 * a:2 * a + 2] - J1[:, :, 2 * a:2 * a + 2]).max(axis=(1, 2))
        assert np.all(err <= 1e-13 * rows), (a, (err / rows).max())
        assert np.abs(F0[a::2] - F1[a::2]).max() <= 1e-13 * np.abs(F1[a::2]).max()
    np.testing.assert_allclose(m0, m1, rtol=1e-14, atol=0)
