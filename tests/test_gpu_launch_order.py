"""Kernels launched with programmatic dependent launch read what their predecessor wrote (pdl_begin): also loads
that stand first in a kernel, without any condition, and that the compiler may take for constant."""
import ctypes
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker deselects these on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1905_08890_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "gr_internal.cuh"

namespace gr {
std::atomic<long long> g_launches{0};
namespace {

// writes v to all cnt words some 20 us after it could start
__global__ void k_write(unsigned *out, int cnt, unsigned v)
{
    pdl_begin();
    for (int k = 0; k < 20; k++) __nanosleep(1000);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x) out[t] = v;
}

// one word for all threads, as a list's length is read
__global__ void k_uniform(const unsigned *__restrict__ in, const unsigned *__restrict__ len, unsigned cap,
                          unsigned *__restrict__ out)
{
    pdl_begin();
    const unsigned n = min(*len, cap);
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) out[t] = in[t] + n;
}

// a word per thread, no bounds check
__global__ void k_each(const unsigned *__restrict__ in, unsigned *__restrict__ out)
{
    pdl_begin();
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    out[t] = in[t] + __ldg(in + (t ^ 1u));
}

// a vector per thread and one word for all, through shared memory
__global__ void k_vector(const float4 *__restrict__ in, const unsigned *__restrict__ one, float4 *__restrict__ out)
{
    pdl_begin();
    __shared__ unsigned s;
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, w = *one;
    float4 v = in[t];
    if (threadIdx.x == 0) s = w;
    __syncthreads();
    v.x += __uint_as_float(s);
    out[t] = v;
}

}  // namespace
}  // namespace gr

// rounds of (write, read); bad[k]: wrong words of reader k
extern "C" int run(int rounds, unsigned *in, unsigned *out, int cnt, unsigned *host, unsigned *bad, void *stream)
{
    using namespace gr;
    cudaStream_t st = (cudaStream_t)stream;
    const int B = 128, G = cnt / B;
    for (int k = 0; k < 3; k++) bad[k] = 0;
    for (int r = 1; r <= rounds; r++)
        for (int k = 0; k < 3; k++) {
            // a length of cnt - r, and float 2 r
            const unsigned v = k == 0 ? cnt - r : (k == 1 ? r * 7u : 0x3f800000u + r);
            GR_LAUNCH(k_write, 32, B, st, in, cnt, v);
            if (k == 0) GR_LAUNCH(k_uniform, 4, B, st, in, in, (unsigned)cnt, out);
            else if (k == 1) GR_LAUNCH(k_each, G, B, st, in, out);
            else GR_LAUNCH(k_vector, G / 4, B, st, (const float4 *)in, in, (float4 *)out);
            if (cudaMemcpyAsync(host, out, cnt * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return 1;
            if (cudaStreamSynchronize(st) != cudaSuccess) return 2;
            for (int t = 0; t < cnt; t++) {
                unsigned want = 2 * v;
                if (k == 0) {
                    if ((unsigned)t >= v) continue;
                } else if (k == 2) {
                    float f;
                    memcpy(&f, &v, 4);
                    f = t % 4 == 0 ? f + f : f;
                    memcpy(&want, &f, 4);
                }
                bad[k] += host[t] != want;
            }
        }
    return cudaGetLastError() == cudaSuccess ? 0 : 3;
}
"""


def test_first_loads_wait_for_the_previous_kernel(tmp_path):
    cu, so = tmp_path / "order.cu", tmp_path / "liborder.so"
    cu.write_text("#include <cstring>\n" + SOURCE)
    subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-I", _build.CSRC, "-shared", str(cu), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    cnt = 4096
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        buf = torch.zeros((2, cnt), dtype=torch.int32, device="cuda")
    stream.synchronize()
    host = torch.zeros(cnt, dtype=torch.int32).pin_memory()
    bad = (ctypes.c_uint * 3)()
    assert lib.run(50, ctypes.c_void_p(buf[0].data_ptr()), ctypes.c_void_p(buf[1].data_ptr()), cnt,
                   ctypes.c_void_p(host.data_ptr()), bad, ctypes.c_void_p(stream.cuda_stream)) == 0
    assert list(bad) == [0, 0, 0]
