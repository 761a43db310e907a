"""A cycle queued before its predecessor's norm is read leaves no trace when that norm ends the solve.

With profile set every norm is read before the next cycle is queued, so both ways have to give the same cycles,
residuals, cell counts and fields.  A checkerboard source is such a case: the error that one red-black sweep leaves
is a constant, so that a single V-cycle takes the residual from 1 to rounding.
"""
import ctypes
import math

import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


def _checkerboard(ctx, n, amplitude):
    src = ctx.new_sources()
    i = torch.arange(n, device="cuda")
    sign = 1.0 - 2.0 * ((i[:, None, None] + i[None, :, None] + i[None, None, :]) % 2).to(torch.float64)
    for k in gr.SOURCES:
        src[k].fill_(synth.RHO_BAR if k == "s0" else 0.0)
    src["sx"].copy_(amplitude * sign)
    return src


def _solve(ctx, src, **kw):
    fld = ctx.initial_fields()
    rep = ctx.solve(src, fld, rho_hat=synth.RHO_BAR, allow_noconv=True, **kw)
    torch.cuda.synchronize()
    return fld, rep


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_df"])
@pytest.mark.parametrize("n", [16, 64, 128])
def test_one_cycle_is_enough(n, prec):
    ctx = gr.Context(n)
    src = _checkerboard(ctx, n, 1e-3 * synth.RHO_BAR)
    fld, rep = _solve(ctx, src, prec=prec, tol=1e-6)
    ref, want = _solve(ctx, src, prec=prec, tol=1e-6, profile=True)
    assert want["cycles"][gr.GR_VX] == 1  # the case is one
    for k in ("cycles", "cell_updates"):
        assert rep[k] == want[k], k
    # the double-float norms are FP32 sums over threads, in an order that alternates from call to call
    assert rep["res"] == pytest.approx(want["res"], rel=1e-4)
    for k in gr.FIELDS:
        assert torch.equal(fld[k], ref[k]), k
    ctx.close()


def test_a_residual_that_overflows_stops_where_it_was_seen():
    """An FP64 residual beyond FP32's range makes the FP32 correction infinite in the first cycle: the call ends
    after that cycle with its residual, whichever way the norms are read."""
    ctx = gr.Context(32)
    src = _checkerboard(ctx, 32, 1e39)
    reps = []
    for profile in (False, True):
        fld = ctx.initial_fields()
        opts = gr.make_opts(prec="mixed", tol=1e-6, rho_hat=synth.RHO_BAR, profile=profile)
        s, f, r = gr.make_sources(src), gr.make_fields(fld), gr.gr_report()
        st = gr.lib().gr_solve_constraints(ctx.h, ctypes.byref(s), ctypes.byref(f), ctypes.byref(opts), ctypes.byref(r))
        assert st == gr.GR_ERR_NONFINITE
        reps.append(r)
    torch.cuda.synchronize()
    assert reps[1].cycles[gr.GR_VX] == 1
    assert list(reps[0].cycles) == list(reps[1].cycles) and reps[0].cell_updates == reps[1].cell_updates
    assert math.isnan(reps[0].res[gr.GR_VX]) == math.isnan(reps[1].res[gr.GR_VX])
    ctx.close()
