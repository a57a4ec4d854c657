"""FP64 levels: a row's sum over its blocks is two sums, of the products with p_w and
with S_n, each a chain of multiply-adds in stencil order, added at the end (half the
chain of one sum through both, and a smaller error).  The residual b - A x of a coarse
level equals, to the last bit, that sum emulated in exact arithmetic with one rounding
per operation, from the exported operator (shift 1, so that shift M - J has one
rounding whatever the compiler fuses); plain and small forms alike."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2506_04763_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
rf = pytest.importorskip("paper_2506_04763_gb300")


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _residual(dim, m, A, b, x):
    out = np.empty_like(b)
    offs = [(dx, dy, dz) for dz in ((-1, 0, 1) if dim == 3 else (0,)) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    for v in range(m[0] * m[1] * m[2]):
        i, j, k = v % m[0], v // m[0] % m[1], v // (m[0] * m[1])
        for h in (0, 1):
            s, t = 0.0, 0.0
            for q, (dx, dy, dz) in enumerate(offs):
                if 0 <= i + dx < m[0] and 0 <= j + dy < m[1] and 0 <= k + dz < m[2]:
                    w = v + dx + m[0] * (dy + m[1] * dz)
                    s = _fma(float(A[v, q, 2 * h]), float(x[2 * w]), s)
                    t = _fma(float(A[v, q, 2 * h + 1]), float(x[2 * w + 1]), t)
            out[2 * v + h] = b[2 * v + h] - (s + t)
    return out


@pytest.mark.parametrize("small", ["0", "40000"])
@pytest.mark.parametrize("n", [(9, 9, 9), (17, 9, 1)])
def test_level_residual_is_two_sums_of_multiply_adds(n, small, monkeypatch):
    import __graft_entry__ as G
    G.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    monkeypatch.setenv("RF_SMALL_NV", small)
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 57)
    g = rf.Grid(prob)
    g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
    g.gmg_setup([1.0], rf.gmg_opts(3, "jacobi", precision="fp64"))
    A, m = g.export_level(1, 0)
    m = [int(t) for t in m]
    nv = m[0] * m[1] * m[2]
    b, x = np.random.default_rng(9).standard_normal((2, 2 * nv))
    got = g.apply(rf.RF_OP_RESIDUAL, 1, 0, b, x, out_len=2 * nv)
    g.close()
    assert np.array_equal(got, _residual(dim, m, np.asarray(A).reshape(nv, -1, 4), b, x))
