"""The deposit over tiles (deposit_tiles.cu) against FP64 index_add.

Bar: 1e-13 of each array's largest value, as for the direct kernels (a product
is off by about 2^-52 of the largest charge of its block, and a cell takes at most a few
thousand of them here).
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402

N = 128


def _particles(npart, L, seed, spread=1.0, v=0.3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = (torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64) * spread) * L
    u = torch.randn((3, npart), generator=g, device="cuda", dtype=torch.float64) * v
    return x, u * torch.tensor([[1.0], [1e-6], [30.0]], device="cuda", dtype=torch.float64)


def _reference(L, x, u, mass, psi=None):
    t = x * (N / L) - 0.5
    fl = torch.floor(t)
    fr, lo = t - fl, fl.to(torch.int64)
    corners = []
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                at = [(lo[d] + s) % N for d, s in enumerate((a, b, c))]
                w = 1.0
                for d, s in enumerate((a, b, c)):
                    w = w * (fr[d] if s else 1.0 - fr[d])
                corners.append(((at[0] * N + at[1]) * N + at[2], w))
    u2 = u.square().sum(0)
    ps = 1.0 if psi is None else sum(w * psi.reshape(-1)[at] for at, w in corners)
    W = torch.sqrt(1.0 + u2 / ps ** 4)
    q = mass * (N / L) ** 3
    out = {}
    for k, v in zip(gr.SOURCES, (q * W, q * u[0], q * u[1], q * u[2], q * u2 / W)):
        o = torch.zeros(N ** 3, device="cuda", dtype=torch.float64)
        for at, w in corners:
            o.index_add_(0, at, v * w)
        out[k] = o.reshape(N, N, N)
    return out


def _run(ctx, x, u, mass, psi=None):
    src = ctx.deposit(x, u, mass) if psi is None else ctx.deposit_metric(x, u, mass, psi)
    torch.cuda.synchronize()
    return src


@pytest.mark.parametrize("metric", [False, True])
@pytest.mark.parametrize("L", [1.0, 0.7])
def test_matches_index_add(L, metric):
    """Uniform particles with a crowd in one cell (several items of one tile),
    others outside the box on both sides, velocities of very different sizes."""
    npart = (2 if metric else 1) * N ** 3 + 77
    x, u = _particles(npart, L, 5)
    x[:, :5000] = x[:, :1] + 1e-9 * L * torch.rand((3, 5000), device="cuda", dtype=torch.float64)
    x[0, 5000:9000] -= 2.0 * L
    x[2, 9000:13000] += 3.0 * L
    x[:, 13000] = torch.tensor([0.0, 0.5 * L / N, L], device="cuda", dtype=torch.float64)
    u[:, 20000:30000] = 0.0
    psi = None
    if metric:
        g = torch.Generator(device="cuda").manual_seed(6)
        psi = 1.0 + 0.2 * torch.rand((N, N, N), generator=g, device="cuda", dtype=torch.float64) - 0.1
    ctx = gr.Context(N, L)
    src = _run(ctx, x, u, 1e-7, psi)
    ref = _reference(L, x, u, 1e-7, psi)
    for k in gr.SOURCES:
        assert (src[k] - ref[k]).abs().max() <= 1e-13 * ref[k].abs().max(), k
    ctx.close()


def test_particles_that_are_not_finite_spoil_their_cells_only():
    """One velocity and one position that are not finite, one velocity of 1e200,
    against the same set without them: cells away from them are unchanged."""
    x, u = _particles(N ** 3, 1.0, 7)
    ctx = gr.Context(N)
    clean = {k: v.clone() for k, v in _run(ctx, x[:, 3:].contiguous(), u[:, 3:].contiguous(), 1e-7).items()}
    x[:, :3] = torch.tensor([[0.25], [0.5], [0.75]], device="cuda", dtype=torch.float64)
    u[:, :3] = 0.0
    u[0, 0], u[1, 1], x[2, 2] = float("inf"), 1e200, float("nan")
    src = _run(ctx, x, u, 1e-7)
    assert not torch.isfinite(src["sx"]).all() and not torch.isfinite(src["s0"]).all()
    for k in gr.SOURCES:
        far = torch.ones((N, N, N), dtype=torch.bool, device="cuda")
        far[30:34, 62:66, :] = False  # the three particles' columns
        d = (src[k] - clean[k])[far]
        assert d.abs().max() <= 1e-13 * clean[k].abs().max(), k
    ctx.close()
