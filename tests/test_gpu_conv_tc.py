"""The tcgen05 convolution at 128^3 against the mma.sync one: with 16 input
channels both sum the same products in the same order, so the activations agree
bit for bit; with 48 the order differs and BF16 roundings may flip."""
import numpy as np
import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


def test_both_tensor_core_paths_give_the_same_layers(monkeypatch):
    """e0a, e0b: equal bits.  d0a (48 -> 16): BF16 roundings, 2^-7 of the value plus 2^-16 of the largest
    (FP32 sums of 1296 products in two orders).  Gradients of the two finest layers (data gradients into 16 and
    48 channels with mask and without): 2^-6 in norm."""
    n = 128
    p = synth.zeldovich(n, 4, 1.0, 0.01, True)
    ctx = gr.Context(n)
    src = ctx.deposit(torch.from_numpy(p.x).cuda(), torch.from_numpy(p.u).cuda(), p.mass)
    tgt = {k: torch.zeros((n, n, n), dtype=torch.float64, device="cuda") for k in gr.FIELDS}
    for k in ("psi", "apsi"):
        tgt[k] += 1.0
    net = gr.Net(n, seed=8)
    net.set_norm([0, 0, 0, 0], [1, 1, 1, 1], np.zeros(10), np.full(10, 1e-3))
    acts, grads = [], []
    for flag in ("1", "0"):
        monkeypatch.setenv("GR_CONV_TC", flag)
        loss, g = net.loss_grad(src, tgt, p.rho_hat, 0.01)
        grads.append(g)
        acts.append({k: net.activation(k) for k in ("e0a", "e0b", "d0a")})
    for k in ("e0a", "e0b"):
        assert np.array_equal(acts[0][k], acts[1][k]), k
    a, b = acts[0]["d0a"], acts[1]["d0a"]
    assert (np.abs(a - b) <= 2.0 ** -7 * np.abs(b) + 2.0 ** -16 * np.abs(b).max()).all()
    for lo in (0, 27 * 256 + 16):  # the first two convolutions
        u, v = grads[0][lo:lo + 27 * 256 + 16], grads[1][lo:lo + 27 * 256 + 16]
        assert np.linalg.norm(u - v) <= 2.0 ** -6 * np.linalg.norm(v)
    net.close()
    ctx.close()
