"""gr_report.cell_updates: the cells that a solve's sweeps relax, the 2^3 level's eight once per cycle."""
import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
@pytest.mark.parametrize("n", [8, 16, 64])
def test_count(n, prec):
    ctx = gr.Context(n)
    x, u, mass = synth.zeldovich_torch(n, 5, 0.5, 0.01, False)
    src = ctx.deposit(x, u, mass)
    rep = ctx.solve(src, ctx.initial_fields(), tol=1e-6, prec=prec, nu1=1, nu2=2, allow_noconv=True)
    levels = [k for k in (4, 8, 16, 32, 64) if k <= n]
    assert sum(rep["cycles"]) > 10
    assert rep["cell_updates"] == sum(rep["cycles"]) * (3 * sum(k ** 3 for k in levels) + 8)
    ctx.close()
