"""Levels of 32^3 and 64^3 of the FP32 correction cycle in one launch per
direction (level_fused.cu) against the separate launches.

GR_COARSE_TAIL=0 takes every level through separate launches.  The two cycles
do the same operations on 32^3 and 64^3; below, the single-block tail also
restricts the black residuals, which are rounding (2^-24 of 6 |e| / h^2).  On
the levels 16^3 and coarser that is at most 2^-24 * 6 * (16 / 2 pi)^2 = 2e-6 of
the right-hand side, amplified by no more than the 10 sums it enters: 1e-4 of a
cycle's change bounds it.
"""
import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("prec", ["mixed_df", "mixed"])
@pytest.mark.parametrize("n", [32, 64, 128])
def test_one_cycle_equals_the_separate_launches(monkeypatch, n, prec):
    out, src = [], None
    for flag in ("1", "0"):
        monkeypatch.setenv("GR_COARSE_TAIL", flag)
        ctx = gr.Context(n)
        if src is None:
            x, u, mass = synth.zeldovich_torch(n, 31, 1.5, 0.01, True)
            src = ctx.deposit(x, u, mass)
        fld = ctx.initial_fields()
        for eq in (gr.GR_VX, gr.GR_PSI, gr.GR_APSI):
            ctx.vcycle(eq, src, fld, prec=prec, rho_hat=synth.RHO_BAR)
        torch.cuda.synchronize()
        out.append(fld)
        ctx.close()
    for k, plain in (("Vx", 0.0), ("psi", 1.0), ("apsi", 1.0)):
        change = (out[1][k] - plain).abs().max()
        assert change > 0
        assert (out[0][k] - out[1][k]).abs().max() <= 1e-4 * change, k
