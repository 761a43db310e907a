"""Positions far outside the box or not finite in the deposit over tiles (deposit_tiles.cu): each such particle
reaches the cells that the direct kernels give it, also where those are inner cells of another tile's.

Bar: 1e-13 of each array's largest value, as for the tiled deposit in general.  A particle of a grid-filling set
carries a cell's mean charge, so one that is lost or misplaced shows at once.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import gr  # noqa: E402

MASS = 1e-7


def _set(N, L, seed, npart):
    """npart particles at speeds of 0.3 (enough of them for the tiles), and the inner cells of tiles, all over the
    box, for 4000 more."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64) * L
    u = 0.3 * torch.randn((3, npart + 4000), generator=g, device="cuda", dtype=torch.float64)
    cell = torch.randint(0, N, (3, 4000), generator=g, device="cuda") // 8 * 8 + 3
    return x, cell, u


def _deposit(ctx, x, u, metric):
    if metric:
        psi = torch.full((ctx.n,) * 3, 1.1, dtype=torch.float64, device="cuda")
        src = ctx.deposit_metric(x.contiguous(), u.contiguous(), MASS, psi)
    else:
        src = ctx.deposit(x.contiguous(), u.contiguous(), MASS)
    torch.cuda.synchronize()
    return {k: src[k].clone() for k in gr.SOURCES}


@pytest.mark.parametrize("metric", [False, True])
@pytest.mark.parametrize("L", [1.0, 0.7])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("sign", [1, -1])
def test_far_positions_are_wrapped(axis, sign, L, metric):
    """2^30 cells and 2^40 cells (a multiple of n) from the box, against the same particles inside it.  The far
    coordinate is that of a cell boundary and a quarter, which is exact at these distances for L = 1; otherwise the
    rounded position is wrapped in exact integer arithmetic for the comparison."""
    from fractions import Fraction

    N = 256 if metric else 128  # the sets that the tiles take
    x, cell, u = _set(N, L, 11 + axis, (3 if metric else 2) * N ** 3 // 2)
    h = L / N
    near = (cell.to(torch.float64) + 0.75) * h
    far = near.clone()
    shift = torch.where(torch.arange(4000, device="cuda") % 2 == 0, 2.0 ** 30, 2.0 ** 40) * sign
    far[axis] = ((cell[axis].to(torch.float64) + 0.75) + shift) * h
    if L != 1.0:  # 1/h and the product are rounded: take t as the kernels form it, one rounding of x * (1/h) - 1/2
        ih = Fraction(float(1.0 / h))
        t = [float(Fraction(v) * ih - Fraction(1, 2)) for v in far[axis].tolist()]
        near[axis] = torch.tensor([float((Fraction(v) % N + Fraction(1, 2)) / ih) for v in t], device="cuda",
                                  dtype=torch.float64)
    ctx = gr.Context(N, L)
    reps = [_deposit(ctx, torch.cat((x, far), 1), u, metric) for _ in range(3)]
    want = _deposit(ctx, torch.cat((x, near), 1), u, metric)
    for k in gr.SOURCES:
        for got in reps:
            assert (got[k] - want[k]).abs().max() <= 1e-13 * want[k].abs().max(), k
    ctx.close()


@pytest.mark.parametrize("L", [1.0, 0.7])
def test_extreme_positions_are_those_of_the_direct_kernel(L):
    """Up to 1e300, infinite and NaN: the tiled deposit equals its finite part plus each such particle on its own
    (one particle takes the direct kernel), including which cells become NaN."""
    N = 128
    x, _, u = _set(N, L, 21, N ** 3)
    u = u[:, : x.shape[1]]
    h = L / N
    inf, nan = float("inf"), float("nan")
    far = [2.0 ** 30 * h, -(2.0 ** 31 + 5.25) * h, (2.0 ** 51 + 3.5) * h, 2.0 ** 52 * h, -(2.0 ** 53 + 2) * h,
           2.0 ** 62 * h, 2.0 ** 63 * h, -(2.0 ** 63) * h, 1e300, -1e300, inf, -inf, nan]
    xf = torch.full((3, len(far)), 0.0, device="cuda", dtype=torch.float64)
    for i, v in enumerate(far):
        xf[:, i] = (torch.tensor([3, 60, 91], device="cuda") + 0.75 + 8 * (i % 4)) * h
        xf[i % 3, i] = v
    uf = 0.1 * torch.ones_like(xf)
    ctx = gr.Context(N, L)
    want = _deposit(ctx, x, u, False)
    for i in range(len(far)):
        one = _deposit(ctx, xf[:, i : i + 1], uf[:, i : i + 1], False)
        for k in gr.SOURCES:
            want[k] += one[k]
    for _ in range(3):
        got = _deposit(ctx, torch.cat((x, xf), 1), torch.cat((u, uf), 1), False)
        for k in gr.SOURCES:
            bad = ~torch.isfinite(want[k])
            assert bad.any() and torch.equal(bad, ~torch.isfinite(got[k])), k
            assert (got[k] - want[k])[~bad].abs().max() <= 1e-13 * want[k][~bad].abs().max(), k
    ctx.close()
