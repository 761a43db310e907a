"""The kernels that sum weight gradients over the voxels (head and last 3^3
convolution) against plain FP64 sums over the network's own activations, on
grids that give every block one box of voxels, an uneven share, and many."""
import numpy as np
import pytest

from paper_1905_08890_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402


@pytest.mark.parametrize("n", [32, 64, 128])
def test_last_layer_gradients_match_fp64_sums(n):
    """dout = 2 (out - t) / (10 nv) in FP32: within 2^-20 of 2 (sum |W||a| + |b| + |t|) / (10 nv);
    the head's sums add at most 2^-18 of their absolute terms.  dy = (a > 0) W^T dout is rounded to
    BF16, so every weight and bias of the convolution is within 2^-8 sum |x||dy| plus the head's part."""
    p = synth.zeldovich(n, 7, 1.0, 0.01, True)
    ctx = gr.Context(n)
    src = ctx.deposit(torch.from_numpy(p.x).cuda(), torch.from_numpy(p.u).cuda(), p.mass)
    rng = torch.Generator(device="cuda").manual_seed(n)
    tgt = {k: 1e-3 * torch.randn((n, n, n), dtype=torch.float64, device="cuda", generator=rng) for k in gr.FIELDS}
    t = torch.stack([tgt[k].reshape(-1) for k in gr.FIELDS], 1) / 1e-3
    for k in ("psi", "apsi"):
        tgt[k] += 1.0
    net = gr.Net(n, seed=3)
    net.set_norm([0, 0, 0, 0], [1, 1, 1, 1], np.zeros(10), np.full(10, 1e-3))
    params = torch.from_numpy(net.get_params()).cuda().double()
    loss, g = net.loss_grad(src, tgt, p.rho_hat, 0.01)
    g = torch.from_numpy(g).cuda().double()
    a = torch.as_tensor(net.activation("d0b")).cuda().double().reshape(-1, 16)
    x = torch.as_tensor(net.activation("d0a")).cuda().double()
    W, b = params[-170:-10].reshape(10, 16), params[-10:]
    c = 2.0 / (10 * n ** 3)
    r = a @ W.T + b - t
    dout = c * r
    dabs = c * (a.abs() @ W.T.abs() + b.abs() + t.abs())
    assert abs(loss - float((r * r).mean())) <= 2.0 ** -12 * float((r * r).mean())
    tiny = 2.0 ** -18
    assert ((g[-170:-10].reshape(10, 16) - dout.T @ a).abs() <= tiny * (dabs.T @ a.abs())).all()
    assert ((g[-10:] - dout.sum(0)).abs() <= tiny * dabs.sum(0)).all()
    on = (a > 0).double()
    dy, dya = on * (dout @ W), on * (dabs @ W.abs())
    tol = 2.0 ** -8 * dy.abs() + tiny * dya
    gw, gb = g[-170 - 16 - 27 * 256:-170 - 16].reshape(27, 16, 16), g[-170 - 16:-170]
    assert ((gb - dy.sum(0)).abs() <= tol.sum(0)).all()
    for tap in range(27):
        off = (1 - tap // 9, 1 - tap // 3 % 3, 1 - tap % 3)
        xs = torch.roll(x, off, dims=(0, 1, 2)).reshape(-1, 16)
        err = (gw[tap] - dy.T @ xs).abs()
        assert (err <= tol.T @ xs.abs()).all(), (tap, float(err.max()))
    net.close()
    ctx.close()
