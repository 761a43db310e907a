"""The deposit over tiles in several passes (deposit_tiles.cu): more particles than its scratch holds at a time, and
host arrays whose chunks go partly over tiles and partly to the direct kernel.

Bar: 1e-13 of each array's largest value, as for one pass (test_gpu_deposit_tiles).
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402

MASS = 1e-7


def _particles(npart, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64)
    return x, 0.3 * torch.randn((3, npart), generator=g, device="cuda", dtype=torch.float64)


def _check(src, n, x, u, psi=None):
    t = x * n - 0.5
    fl = torch.floor(t)
    fr, lo = t - fl, fl.to(torch.int64)
    corners = []
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                at = [(lo[d] + s) % n for d, s in enumerate((a, b, c))]
                w = 1.0
                for d, s in enumerate((a, b, c)):
                    w = w * (fr[d] if s else 1.0 - fr[d])
                corners.append(((at[0] * n + at[1]) * n + at[2], w))
    u2 = u.square().sum(0)
    ps = 1.0 if psi is None else sum(w * psi.reshape(-1)[at] for at, w in corners)
    W = torch.sqrt(1.0 + u2 / ps ** 4)
    q = MASS * float(n) ** 3
    for k, v in zip(gr.SOURCES, (q * W, q * u[0], q * u[1], q * u[2], q * u2 / W)):
        o = torch.zeros(n ** 3, device="cuda", dtype=torch.float64)
        for at, w in corners:
            o.index_add_(0, at, v * w)
        o = o.reshape(n, n, n)
        assert (src[k] - o).abs().max() <= 1e-13 * o.abs().max(), k


@pytest.mark.parametrize("per_cell", [3, 7])
def test_more_particles_than_the_scratch_holds(per_cell):
    n = 128
    x, u = _particles(per_cell * n ** 3 + 77, 51)
    ctx = gr.Context(n)
    src = ctx.deposit(x, u, MASS)
    torch.cuda.synchronize()
    _check(src, n, x, u)
    ctx.close()


def test_more_particles_than_the_scratch_holds_with_the_metric():
    n = 256
    x, u = _particles(3 * n ** 3 + 1, 52)
    psi = 1.0 + 0.1 * torch.sin(6.283185307179586 * torch.arange(n, device="cuda", dtype=torch.float64) / n)
    psi = (psi[:, None, None] * psi[None, :, None]).expand(n, n, n).contiguous()
    ctx = gr.Context(n)
    src = ctx.deposit_metric(x, u, MASS, psi)
    torch.cuda.synchronize()
    _check(src, n, x, u, psi)
    ctx.close()


def test_host_chunks_over_tiles_and_direct(monkeypatch):
    n, chunk = 128, 2200000
    monkeypatch.setenv("GR_HOST_CHUNK", str(chunk))
    x, u = _particles(2 * chunk + 5000, 53)
    ctx = gr.Context(n)
    src = ctx.deposit(x.cpu().pin_memory(), u.cpu().pin_memory(), MASS)
    torch.cuda.synchronize()
    _check(src, n, x, u)
    ctx.close()
