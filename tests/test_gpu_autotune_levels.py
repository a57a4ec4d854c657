"""The autotuner times candidates only on levels whose kernels have a shape to choose:
the small levels' FP64 and FP32 kernels have one shape, and a choice among seven
timings of the same launch would be noise, kept in the process and in the cache
file.  FP16 storage and levels beyond the small ones are tuned as before, and a line
of the file is still read."""
import json

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


def _tuned(n, levels, smoother, precision, tmp_path, monkeypatch):
    cache = tmp_path / "tune.jsonl"
    monkeypatch.setenv("RF_TUNE_CACHE", str(cache))
    dim = 3 if n[2] > 1 else 2
    prob = I.random_problem(dim, n if dim == 3 else n[:2], 67)
    g = rf.Grid(prob)
    g.assemble(torch.tensor(prob["u0"], device="cuda"), True)
    g.gmg_setup([0.1], rf.gmg_opts(levels, smoother, precision=precision, autotune=True))
    g.close()
    lines = cache.read_text().splitlines() if cache.exists() else []
    return [json.loads(t)["key"].split("|")[1] for t in lines]


# (sizes that no other test tunes: a choice is made once per process)
@pytest.mark.parametrize("smoother,precision,n", [("gs8", "fp64", (29, 13, 17)), ("gs8", "fp32", (29, 13, 21)),
                                                  ("jacobi", "fp64", (29, 13, 25)), ("jacobi", "fp32", (29, 17, 13))])
def test_small_levels_are_not_timed(smoother, precision, n, tmp_path, monkeypatch):
    assert _tuned(n, 3, smoother, precision, tmp_path, monkeypatch) == []


def test_other_levels_are(tmp_path, monkeypatch):
    assert _tuned((29, 17, 21), 3, "gs8", "fp16", tmp_path, monkeypatch) == ["29x17x21"]
    assert _tuned((45, 37, 29), 3, "gs8", "fp32", tmp_path, monkeypatch)[1:] == ["45x37x29"]
