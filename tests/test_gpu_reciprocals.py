"""recip64 and rsqrt64 (gr_internal.cuh), which stand for FP64 divisions and square roots, against those.

Bars: after two Newton steps the estimate's 2^-20 has become 2^-80 and what is left are the last step's roundings: of
x r to 1 - x r (exact but for 2^-53 of a small number) and of the result: one unit in the last place.  rsqrt64: the
estimate is good to 2^-21, so that the third-order step's error is below 2^-62; e = 1 - a y^2 is off by 2^-53 from the
rounding of a y, half of which enters y, next to the result's rounding: two units.  Zeros, infinities, NaN and
operands with a subnormal reciprocal or value are those of the division, bit for bit.
"""
import ctypes
import math
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "gr_internal.cuh"
__global__ void k(int which, int cnt, const double *x, double *y)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) y[t] = which ? gr::rsqrt64(x[t]) : gr::recip64(x[t]);
}
extern "C" int run(int which, int cnt, const double *x, double *y)
{
    k<<<(cnt + 255) / 256, 256>>>(which, cnt, x, y);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("reciprocals")
    (d / "r.cu").write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-I", _build.CSRC, "-shared", str(d / "r.cu"), "-o",
                    str(d / "libr.so")], check=True)
    lib = ctypes.CDLL(str(d / "libr.so"))

    def call(which, x):
        x = torch.as_tensor(x, dtype=torch.float64).cuda()
        y = torch.empty_like(x)
        assert lib.run(which, x.numel(), ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr())) == 0
        return x.cpu().numpy(), y.cpu().numpy()

    return call


def _mantissas(seed, cnt=1 << 20):
    r = np.random.default_rng(seed)
    return np.concatenate([1.0 + r.random(cnt), 1.0 + 2.0 ** -52 * np.arange(64), 2.0 - 2.0 ** -52 * np.arange(1, 65)])


def test_reciprocal_to_one_unit(run):
    m = _mantissas(1)
    for e in (-1021, -300, -30, -1, 0, 1, 30, 300, 1021):
        x, y = run(0, np.ldexp(m, e) * np.where(np.arange(m.size) % 3 == 0, -1.0, 1.0))
        want = 1.0 / x
        assert (np.abs(y - want) <= np.spacing(np.abs(want))).all(), e


def test_reciprocal_of_the_rest(run):
    tiny = 5e-324
    x = [0.0, -0.0, math.inf, -math.inf, math.nan, tiny, -tiny, 1e-310, 2.0 ** -1022, 2.0 ** -1023, 2.0 ** 1022,
         1.7e308, -2.0 ** 1023]
    x, y = run(0, x)
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    assert ((y == want) | (np.isnan(y) & np.isnan(want))).all() and (np.signbit(y) == np.signbit(want))[~np.isnan(x)].all()


def test_inverse_root_to_two_units(run):
    m = _mantissas(2)
    for e in (0, 1, 2, 3, 30, 31, 119, 120, 400, 1000):
        x, y = run(1, np.ldexp(m, e))
        want = 1.0 / np.sqrt(x.astype(np.longdouble))
        assert (np.abs(y - want) <= 2.0 * np.spacing(want.astype(np.float64))).all(), e
    x, y = run(1, [1.0, math.inf, math.nan])
    assert y[0] == 1.0 and y[1] == 0.0 and math.isnan(y[2])
