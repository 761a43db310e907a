"""FP64 V-cycles whose levels of 16^3 and coarser run in one cluster launch
(fp64_tail.cu) against the separate launches (GR_COARSE_TAIL=0).

Both do the same cycle; sums are paired differently, reciprocals differ by a
rounding and the cluster drops the black residuals, which are rounding: 2^-53
of 6 |u| / h^2, on 32^3 at most 2^-53 * 6 * (32 / 2 pi)^2 = 2e-14 of the
right-hand side, in sums of up to 100 terms: 1e-11 of a cycle's change bounds
the difference.
"""
import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 0), (0, 3)])
@pytest.mark.parametrize("n", [4, 8, 16, 32])
def test_one_cycle_equals_the_separate_launches(monkeypatch, n, nu1, nu2):
    out, src = [], None
    for flag in ("1", "0"):
        monkeypatch.setenv("GR_COARSE_TAIL", flag)
        ctx = gr.Context(n)
        if src is None:
            x, u, mass = synth.zeldovich_torch(n, 33, 1.5, 0.1, True)
            src = ctx.deposit(x, u, mass)
        fld = ctx.initial_fields()
        for eq in (gr.GR_VX, gr.GR_VY, gr.GR_VZ, gr.GR_U, gr.GR_PSI, gr.GR_APSI):
            ctx.vcycle(eq, src, fld, prec="fp64", rho_hat=synth.RHO_BAR, nu1=nu1, nu2=nu2)
        torch.cuda.synchronize()
        out.append(fld)
        ctx.close()
    for k, plain in (("Vx", 0.0), ("U", 0.0), ("psi", 1.0), ("apsi", 1.0)):
        change = (out[1][k] - plain).abs().max()
        assert change > 0
        # psi and alpha psi are returned with 1 added: their rounding is that of 1
        assert (out[0][k] - out[1][k]).abs().max() <= 1e-11 * change + 2.0 ** -52, k
