"""Relative accuracy of every cell of the tiled deposit (deposit_tiles.cu), also where a cell's charges are small
beside those of other cells of its tile.

A sum is good to 2^-46 of the sum of its charges' magnitudes, as the direct kernels' double-float products are.  The
bar is 2^-44: the FP64 additions of the comparison and of the atomics come to it, up to 2^-53 per addition of a
cell's few hundred (with a crowd of 6000 in one cell: 6000 x 2^-53 / 2 = 2^-41.5 at worst, 2^-47 as a random walk).
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402

N = 128
MASS = 3e-7


def _cells(x, u, psi=None, N=N):
    """The five sums and the sums of their terms' magnitudes, in FP64."""
    t = x * N - 0.5
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
    q = MASS * float(N) ** 3
    out = {}
    for k, v in zip(gr.SOURCES, (q * W, q * u[0], q * u[1], q * u[2], q * u2 / W)):
        o, m = (torch.zeros(N ** 3, device="cuda", dtype=torch.float64) for _ in range(2))
        for at, w in corners:
            o.index_add_(0, at, v * w)
            m.index_add_(0, at, (v * w).abs())
        out[k] = (o.reshape(N, N, N), m.reshape(N, N, N))
    return out


def _check(x, u, psi=None, N=N):
    ctx = gr.Context(N)
    src = ctx.deposit(x, u, MASS) if psi is None else ctx.deposit_metric(x, u, MASS, psi)
    torch.cuda.synchronize()
    want = _cells(x, u, psi, N)
    for k in gr.SOURCES:
        o, m = want[k]
        err = (src[k] - o).abs()
        worst = torch.nan_to_num(err / m, nan=0.0).max().item()
        assert (err <= 2.0 ** -44 * m).all(), (k, worst * 2.0 ** 44)
    ctx.close()


def _uniform(npart, v, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64)
    return x, v * torch.randn((3, npart), generator=g, device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("v", [0.01, 30.0])
def test_particles_of_one_temperature(v):
    """Two particles per cell: voids and cells grazed by a single cloud."""
    _check(*_uniform(2 * N ** 3, v, 41))


@pytest.mark.parametrize("fast", [1.0, 1e6])
def test_slow_cells_beside_fast_particles(fast):
    """|u| of 1e-9 everywhere but for one particle in 800: most of s_x and s_z is added in FP64, and more
    particles than the list of those takes."""
    x, u = _uniform(2 * N ** 3 + 5, 1e-9, 42)
    u[0, ::800] = fast
    u[2, 400::800] = -fast
    _check(x, u)


def test_half_at_rest():
    x, u = _uniform(2 * N ** 3, 0.3, 43)
    u[:, x[0] < 0.47] = 0.0
    _check(x, u)


def test_crowds_with_random_velocities():
    """Several blocks per tile, thousands of particles in a cell."""
    x, u = _uniform(2 * N ** 3, 0.1, 44)
    for i in range(40):
        s = slice(6000 * i, 6000 * (i + 1))
        x[:, s] = (x[:, 6000 * i : 6000 * i + 1] + (1.5 / N if i % 2 else 1e-7) * x[:, s]) % 1.0
    _check(x, u)


def test_grazing_clouds():
    """A lattice at the centres of every other plane of cells, displaced by 1e-7 of a cell: the planes between
    hold weights of 1e-7 only, their edges and corners 1e-14 and 1e-21."""
    i = torch.arange(N // 2, device="cuda", dtype=torch.float64) * 2 + 0.5
    x = torch.stack(torch.meshgrid(i, i, i, indexing="ij")).reshape(3, -1).repeat(1, 16)
    g = torch.Generator(device="cuda").manual_seed(45)
    x = (x + 1e-7 * torch.rand(x.shape, generator=g, device="cuda", dtype=torch.float64)) / N
    _check(x.contiguous(), 0.1 * torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64))


def test_with_the_metric():
    n = 256
    x, u = _uniform(3 * n ** 3 // 2 + 3, 1e-7, 46)
    u[1, ::4000] = 0.5
    g = torch.Generator(device="cuda").manual_seed(47)
    psi = 0.8 + 0.4 * torch.rand((n, n, n), generator=g, device="cuda", dtype=torch.float64)
    _check(x, u, psi, n)
