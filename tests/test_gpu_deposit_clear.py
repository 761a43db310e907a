"""A deposit overwrites its five output arrays, whatever was in them."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("n", [4, 8, 64])
@pytest.mark.parametrize("npart", [0, 1])
def test_outputs_are_cleared(n, npart):
    """One resting particle at a cell centre: s0 is its charge there, every other value exactly zero."""
    ctx = gr.Context(n)
    src = {k: torch.full((n, n, n), float("nan"), dtype=torch.float64, device="cuda") for k in gr.SOURCES}
    x = torch.full((3, npart), 1.5 * ctx.L / n, dtype=torch.float64, device="cuda")
    ctx.deposit(x, torch.zeros_like(x), 2.0, src)
    for k in gr.SOURCES:
        want = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
        if npart and k == "s0":
            want[1, 1, 1] = 2.0 * (n / ctx.L) ** 3
        assert ((src[k] - want).abs() <= 2.0 ** -40 * want.abs().max()).all(), k
    ctx.close()
