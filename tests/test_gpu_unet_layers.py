"""Upsampling and head on grids of several blocks per kernel (the 32^3 network's
grids fit in few), against FP64 on the network's own activations."""
import numpy as np
import pytest

from oracle import unet_ref
from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("n", [32, 64])
def test_upsampling_and_head_match_fp64(n):
    """Upsampling: FP32 sums rounded to BF16, within 2^-8 of the sum of absolute terms.  Head: FP32 sums of 17
    terms, within 2^-19 of their absolute sum (and the FP32 de-standardisation, mean 0, deviation 1)."""
    p = synth.zeldovich(n, 9, 1.0, 0.01, True)
    ctx = gr.Context(n)
    src = ctx.deposit(torch.from_numpy(p.x).cuda(), torch.from_numpy(p.u).cuda(), p.mass)
    net = gr.Net(n, seed=6)
    net.set_norm([0, 0, 0, 0], [1, 1, 1, 1], np.zeros(10), np.ones(10))
    out = {k: torch.empty((n, n, n), dtype=torch.float64, device="cuda") for k in gr.FIELDS}
    net.infer(src, out, p.rho_hat, 0.01)
    for lo, cat, c in (("e3b", "cat2", 128), ("d2b", "cat1", 64), ("d1b", "cat0", 32)):
        x = torch.as_tensor(net.activation(lo)).permute(3, 0, 1, 2).unsqueeze(0).double()
        got = net.activation(cat)[..., :c]
        want = unet_ref.up2(x)[0].permute(1, 2, 3, 0).numpy()
        scale = unet_ref.up2(x.abs())[0].permute(1, 2, 3, 0).numpy()
        assert (np.abs(got - want) <= 2.0 ** -8 * scale).all(), lo
    params = net.get_params().astype(np.float64)
    W, b = params[-170:-10].reshape(10, 16), params[-10:]
    a = net.activation("d0b").astype(np.float64)
    for k, name in enumerate(gr.FIELDS):
        got = out[name].cpu().numpy() - (1.0 if k < 2 else 0.0)
        assert (np.abs(got - (a @ W[k] + b[k])) <= 2.0 ** -19 * (a @ np.abs(W[k]) + np.abs(b[k]) + 1e-6)).all(), name
    net.close()
    ctx.close()
