"""The group kernels' quotient by 1 + t against IEEE division: the same bits (the
sign of a zero aside) for ordinary numerators, infinities and not-a-numbers;
within half a last place and 2^-150 for numerators below 2^-90, whose remainder
may be subnormal; divisors at the ends of the mantissa's range.  The device
function is compiled into a small library of its own."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "wave_group.cuh"
namespace empso {
namespace {
__global__ void quotient_kernel(const float4 *n, const float4 *d, float4 *q, int count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float4 a = n[i], b = d[i];
    float2 n01 = lo2(a), n23 = hi2(a);
    n01 = quot2(n01, lo2(b));
    n23 = quot2(n23, hi2(b));
    q[i] = make_float4(n01.x, n01.y, n23.x, n23.y);
}
}
}
extern "C" int probe(const float4 *n, const float4 *d, float4 *q, int count, void *st)
{
    empso::quotient_kernel<<<(count + 127) / 128, 128, 0, (cudaStream_t)st>>>(n, d, q, count);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1905_12795_gb300 import build as b
    path = tmp_path_factory.mktemp("quotient")
    (path / "probe.cu").write_text(SOURCE)
    subprocess.check_call([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared",
                           "-I", b.INCLUDE, "-I", b.CSRC, "-o", str(path / "probe.so"), str(path / "probe.cu")])
    return ctypes.CDLL(str(path / "probe.so"))


def _divisors(rng, n):
    d = (1.0 + rng.random(n) * rng.choice([1e-6, 0.01, 0.3, 5.0, 4000.0], n)).astype(np.float32)
    ends = np.array([1.0, np.nextafter(np.float32(1), np.float32(2)), np.nextafter(np.float32(2), np.float32(1)),
                     np.nextafter(np.float32(4), np.float32(2)), 1.5, 4095.9998], np.float32)
    d[:: 7] = rng.choice(ends, len(d[:: 7]))
    return d


@pytest.mark.parametrize("kind", ["ordinary", "front", "special"])
def test_equals_division(probe, kind):
    rng = np.random.default_rng(len(kind))
    n = 1 << 22
    d = _divisors(rng, n)
    lo, hi = {"ordinary": (-90, 127), "front": (-149, -80), "special": (-149, 127)}[kind]
    num = (rng.choice([-1.0, 1.0], n) * (1.0 + rng.random(n)) * np.exp2(rng.uniform(lo, hi, n).round())).astype(np.float32)
    num[rng.random(n) < 0.02] = 0.0
    num[rng.random(n) < 0.02] = -0.0
    if kind == "special":
        for v in (np.inf, -np.inf, np.nan, np.finfo(np.float32).max):
            num[rng.random(n) < 0.02] = v
        num[: n // 4] = 0.0
    with np.errstate(all="ignore"):
        want = num / d
    a, b = torch.tensor(num, device="cuda"), torch.tensor(d, device="cuda")
    q = torch.zeros_like(a)
    st = torch.cuda.current_stream().cuda_stream
    assert probe.probe(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), ctypes.c_void_p(q.data_ptr()), n // 4,
                       ctypes.c_void_p(st)) == 0
    got = q.cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    wrong = ~nan & (got != want)
    small = np.abs(num) < 2.0 ** -90
    with np.errstate(all="ignore"):
        off = np.abs(got.astype(np.float64) - num.astype(np.float64) / d.astype(np.float64))
    wrong &= ~(small & (off <= 0.5 * np.spacing(np.abs(got)).astype(np.float64) * (1 + 2.0 ** -20) + 2.0 ** -150))
    bad = np.flatnonzero(wrong)
    assert bad.size == 0, (bad.size, num[bad[:4]], d[bad[:4]], got[bad[:4]], want[bad[:4]])
