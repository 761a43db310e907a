"""Cells and weights of the particle update at the edges of their integer forms.

In fields linear in one coordinate away from the wrap the interpolation is
exact, so a drift with alpha = psi = 1 moves a particle by -dt beta(x) with beta
the shift at the particle: positions on cell centres and faces, in the first
half cell (the FP64 form), outside the box, and a box side that is no power of two.
Bar: FP32 interpolation, 8 roundings of the largest shift plus the step's
change of position.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("offset", [0, 1])  # fields on and off 16-byte boundaries
@pytest.mark.parametrize("L", [1.0, 4.0, 0.7])
@pytest.mark.parametrize("n", [4, 32])
def test_drift_in_a_linear_shift(n, L, offset):
    h = L / n
    ctx = gr.Context(n, L)
    dev = {"dtype": torch.float64, "device": "cuda"}
    fld = {}
    for k in gr.FIELDS:
        fld[k] = torch.zeros(n ** 3 + 2, **dev)[offset:offset + n ** 3].view(n, n, n)
    fld["psi"].fill_(1.0)
    fld["apsi"].fill_(1.0)
    centre = (torch.arange(n, **dev) + 0.5) * h
    fld["Bx"] += 0.3 * centre.reshape(n, 1, 1) / L
    fld["Bz"] += 0.2 * centre.reshape(1, 1, n) / L
    # inside the linear range of the periodic grid: half a cell from either end
    t = torch.cat([torch.linspace(0.5, n - 0.5, 257, **dev), torch.arange(1, n, **dev), torch.arange(0.5, n, 1.0, **dev)])
    t = t.clamp(0.5, n - 0.5)
    x = torch.stack([t * h, t.flip(0) * h, t * h]).contiguous()
    x[0, ::3] -= L  # the same place outside the box
    x[2, ::5] += 2.0 * L
    u = torch.zeros_like(x)
    x0, dt = x.clone(), 0.01 * h
    ctx.particle_update(x, u, fld, dt, gr.GR_DRIFT)
    torch.cuda.synchronize()
    place = torch.stack([t * h, t.flip(0) * h, t * h])
    want = place - dt * torch.stack([0.3 * place[0] / L, torch.zeros_like(t), 0.2 * place[2] / L])
    d = (x - want + 0.5 * L) % L - 0.5 * L
    assert d.abs().max() <= 8 * 2.0 ** -24 * 0.3 * dt + 2.0 ** -50 * x0.abs().max()
    assert (u == 0.0).all()
    ctx.close()
