"""The psi equation's 2^3 level in the FP64 cluster launch (fp64_tail.cu) where Newton's method, started at the
restricted guess, would step through psi = 0 to a root with negative conformal factors: the cycle equals that of the
separate launches, whose red-black sweeps stay on the positive branch.

A guess of 0.5 to 2.5 at high background densities, AA = 0; the seeds are the first four for which an emulation of
both cycles in numpy found the negative root.  Bar: that of test_gpu_fp64_tail.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("seed", [810, 1182, 2158, 4339])
def test_positive_branch(monkeypatch, seed):
    n = 4
    rng = np.random.default_rng(seed)
    rho = 10 ** rng.uniform(0.5, 2.5)
    s0 = rho * 10 ** rng.uniform(-2, 0.5) * np.exp(2.0 * rng.normal(size=(n,) * 3))
    guess = np.maximum(rng.uniform(0.5, 1.5) + 0.3 * rng.normal(size=(n,) * 3), -0.5)
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("GR_COARSE_TAIL", flag)
        ctx = gr.Context(n)
        src = ctx.new_sources()
        for k in gr.SOURCES:
            src[k].zero_()
        src["s0"].copy_(torch.from_numpy(s0))
        fld = ctx.initial_fields()
        fld["psi"].copy_(torch.from_numpy(1.0 + guess))
        ctx.vcycle(gr.GR_PSI, src, fld, prec="fp64", rho_hat=rho)
        torch.cuda.synchronize()
        out.append(fld["psi"])
        ctx.close()
    assert (out[1] > 0).all()
    change = (out[1] - 1.0 - torch.from_numpy(guess).cuda()).abs().max()
    assert (out[0] - out[1]).abs().max() <= 1e-11 * change + 2.0 ** -52
