"""The push kernels' own reciprocals (csrc/quotients.cuh), called directly from a
small kernel: every FP32 binade from 1 to the overflow for 2 / x (0.501 ulp: one
Newton step on an approximation within 2^-23 leaves 2^-46 and one rounding) and
1 / sqrt(x) (CUDA's rsqrtf, bit for bit), and FP64 quotients against CUDA's
division, bit for bit."""
import ctypes
import subprocess

import numpy as np
import pytest

from _gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu

PROBE = """
#include "quotients.cuh"
__global__ void f32(const float* x, int n, float* two_over, float* rs, float* rs_cuda)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    two_over[i] = pic::two_over_ge1(x[i]);
    rs[i] = pic::rsqrt_ge1(x[i]);
    rs_cuda[i] = rsqrtf(x[i]);
}
__global__ void f64(const double* a, const double* g, int n, double* q, double* q_cuda)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const pic::Over64 over(g[i]);
    q[i] = over(a[i]);
    q_cuda[i] = a[i] / g[i];
}
extern "C" int run_f32(const float* x, int n, float* a, float* b, float* c)
{
    f32<<<(n + 255) / 256, 256>>>(x, n, a, b, c);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_f64(const double* a, const double* g, int n, double* q, double* r)
{
    f64<<<(n + 255) / 256, 256>>>(a, g, n, q, r);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    require_gpu()
    from paper_1606_02862_gb300 import build as B

    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    subprocess.run([B.nvcc(), *B._flags(), "-shared", "-o", str(d / "probe.so"), str(d / "probe.cu"), "-lcudart"], check=True)
    return ctypes.CDLL(str(d / "probe.so"))


def _call(fn, ins, outs):
    import torch

    ts = [torch.from_numpy(a).cuda() for a in ins]
    os = [torch.empty_like(ts[0]) for _ in range(outs)]
    p = [ctypes.c_void_p(t.data_ptr()) for t in ts + os]
    torch.cuda.synchronize()
    assert fn(*p[:len(ts)], ts[0].numel(), *p[len(ts):]) == 0
    return [o.cpu().numpy() for o in os]


def test_fp32(probe):
    rng = np.random.default_rng(1)
    m = 1.0 + rng.integers(0, 1 << 23, (128, 1 << 14)) * 2.0 ** -23
    x = (m * 2.0 ** np.arange(128.0)[:, None]).reshape(-1).astype(np.float32)
    x[:4] = 1.0, np.finfo(np.float32).max, np.inf, np.nextafter(np.float32(1), np.float32(2))
    two_over, rs, rs_cuda = _call(probe.run_f32, [x], 3)
    assert two_over[2] == 0.0 and rs[2] == 0.0
    assert np.array_equal(rs, rs_cuda)
    k = np.isfinite(x)
    want = 2.0 / x[k].astype(np.float64)
    ulp = np.maximum(2.0 ** (np.floor(np.log2(want)) - 23.0), 2.0 ** -149)
    err = np.abs(two_over[k].astype(np.float64) - want) / ulp
    # a result below 2^-126 (x above 2^127) is rounded a second time, to its coarser ulp
    assert np.max(err[want >= 2.0 ** -126]) <= 0.501
    assert np.max(err) <= 1.0


def test_fp64(probe):
    rng = np.random.default_rng(2)
    n = 1 << 21
    a = rng.normal(0, 1, n) * 10.0 ** rng.uniform(-200, 200, n)
    a[: n // 2] = rng.normal(0, 1, n // 2) * 10.0 ** rng.uniform(-12, 3, n // 2)
    g = np.sqrt(1.0 + (rng.normal(0, 1, n) * 10.0 ** rng.uniform(-8, 8, n)) ** 2)
    a[:3] = 0.0, 1.0, -1.0
    g[3:6] = 1.0, np.inf, np.nextafter(1.0, 2.0)
    q, want = _call(probe.run_f64, [a, g], 2)
    assert np.array_equal(q, want)
    assert q[4] == 0.0
