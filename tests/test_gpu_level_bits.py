"""level_fused.cu's one launch per direction against the separate kernels it stands for, bit for bit.

The kernels are called through the library's internal C++ interface (gr_internal.cuh), on random data."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "gr_internal.cuh"
using namespace gr;

// e: in the first red pass's values (from_r = 0) and out; the fused launch writes eb, ec, rc, the separate ones e, ec2, rc2
extern "C" int down(int kind, int n, int from_r, float *e, float *eb, const float *r, const float *m, const float *inv,
                    double h2, float *ec, float *rc, float *ec2, float *rc2, const float *cinv, double h2c)
{
    const size_t half = (size_t)n * n * n / 2;
    if (from_r) cudaMemset(e, 0, 2 * half * sizeof(float));
    level_down(kind, n, from_r, e, eb, r, m, inv, h2, 1.0 / h2, ec, rc, cinv, h2c, 0);
    if (from_r) sweep_colour<float>(kind, n, e, r, m, inv, h2, 1.0 / h2, 0.0, 0, 0);
    sweep_colour<float>(kind, n, e, r, m, inv, h2, 1.0 / h2, 0.0, 1, 0);
    sweep_colour<float>(kind, n, e, r, m, inv, h2, 1.0 / h2, 0.0, 0, 0);
    sweep_colour<float>(kind, n, e, r, m, inv, h2, 1.0 / h2, 0.0, 1, 0);
    resid_restrict_red(kind, n, e, r, m, 1.0 / h2, ec2, rc2, h2c > 0 ? cinv : nullptr, h2c, 0);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

// black half eb corrected from ec, four passes; e from the fused launch, e2 (black half given) from the separate ones;
// uh, ul and uh2, ul2: the same with the update of the double-float unknown
extern "C" int up(int kind, int n, float *e, const float *eb, const float *r, const float *inv, const float *ec, double h2,
                  float *e2, float *uh, float *ul, float *uh2, float *ul2)
{
    const size_t half = (size_t)n * n * n / 2;
    level_up(kind, n, e, eb, r, inv, ec, h2, nullptr, nullptr, 0);
    level_up(kind, n, nullptr, eb, r, inv, ec, h2, uh, ul, 0);
    cudaMemcpy(e2 + half, eb, half * sizeof(float), cudaMemcpyDeviceToDevice);
    prolong_add_black(n, e2, ec, 0);
    for (int c = 0; c < 3; c++) sweep_colour<float>(kind, n, e2, r, nullptr, inv, h2, 1.0 / h2, 0.0, c & 1, 0);
    df_black_update(kind, n, e2, r, inv, h2, uh2, ul2, 0);
    sweep_colour<float>(kind, n, e2, r, nullptr, inv, h2, 1.0 / h2, 0.0, 1, 0);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("level")
    so = _build.build()
    (d / "level.cu").write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-I", _build.CSRC, "-shared", str(d / "level.cu"), "-o",
                    str(d / "liblevel.so"), so, "-Xlinker", "-rpath=" + os.path.dirname(so)], check=True)
    return ctypes.CDLL(str(d / "liblevel.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _level(kind, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def rand(cnt):
        return torch.randn(cnt, generator=g, device="cuda", dtype=torch.float32)

    h2 = (1.0 / n) ** 2
    m = 3.0 * torch.rand(n ** 3, generator=g, device="cuda", dtype=torch.float32)
    inv = 1.0 / (6.0 + h2 * m)
    cinv = 1.0 / (6.0 + 4 * h2 * 3.0 * torch.rand(n ** 3 // 8, generator=g, device="cuda", dtype=torch.float32))
    return rand, h2, m, inv, cinv


@pytest.mark.parametrize("kind", [0, 1])  # Poisson, Helmholtz
@pytest.mark.parametrize("n", [32, 64])
@pytest.mark.parametrize("from_r", [True, False])
@pytest.mark.parametrize("first_red", [True, False])
def test_down(lib, kind, n, from_r, first_red):
    rand, h2, m, inv, cinv = _level(kind, n, 61)
    e, r = rand(n ** 3), rand(n ** 3)
    eb = torch.full((n ** 3 // 2,), float("nan"), device="cuda")
    out = [torch.full((n ** 3 // 8,), float("nan"), device="cuda") for _ in range(4)]  # ec, rc, ec2, rc2
    assert lib.down(kind, n, int(from_r), _p(e), _p(eb), _p(r), _p(m), _p(inv), ctypes.c_double(h2), _p(out[0]),
                    _p(out[1]), _p(out[2]), _p(out[3]), _p(cinv), ctypes.c_double(4 * h2 if first_red else 0.0)) == 0
    assert torch.isfinite(eb).all() and torch.equal(eb, e[n ** 3 // 2 :])
    assert torch.equal(out[1], out[3])
    assert torch.equal(out[0], out[2])


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("n", [32, 64])
def test_up(lib, kind, n):
    rand, h2, m, inv, cinv = _level(kind, n, 62)
    eb, r, ec = rand(n ** 3 // 2), rand(n ** 3), rand(n ** 3 // 8)
    e = torch.full((n ** 3,), float("nan"), device="cuda")
    e2 = rand(n ** 3)
    uh = rand(n ** 3)
    ul = uh * 2.0 ** -25
    uh2, ul2 = uh.clone(), ul.clone()
    assert lib.up(kind, n, _p(e), _p(eb), _p(r), _p(inv), _p(ec), ctypes.c_double(h2), _p(e2), _p(uh), _p(ul), _p(uh2),
                  _p(ul2)) == 0
    assert torch.isfinite(e).all() and torch.equal(e, e2)
    assert torch.equal(uh, uh2) and torch.equal(ul, ul2)
