"""The group kernels' bounded wait: a CTA whose group never comes together gives
up after its limit, leaves every instance of the queue not a number (none keeps
an earlier launch's misfit) and records the time-out where there is a status
word.  One CTA of a group of two is launched by itself, by a small library of
its own."""
import ctypes
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "wave_group.cuh"
namespace empso {
namespace {
__global__ void insts_kernel(Inst *insts, int n)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        insts[i] = Inst{};
        insts[i].out = n - 1 - i;
    }
}
__global__ void __launch_bounds__(WAVE_THREADS) lone_kernel(const Inst *insts, int n, int *ws, int *err, double *partial)
{
    group_cta<1, false, false, false>(nullptr, insts, n, 2, ws, nullptr, 0, err, partial);
}
}
}
using namespace empso;
extern "C" int inst_bytes() { return (int)sizeof(Inst); }
extern "C" int ws_bytes() { return (int)wave_ws_bytes(); }
extern "C" int probe(Inst *insts, int n, int *ws, int *err, double *partial, void *st)
{
    insts_kernel<<<1, 32, 0, (cudaStream_t)st>>>(insts, n);
    lone_kernel<<<1, WAVE_THREADS, 0, (cudaStream_t)st>>>(insts, n, ws, err, partial);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1905_12795_gb300 import build as b
    path = tmp_path_factory.mktemp("timeout")
    (path / "probe.cu").write_text(SOURCE)
    subprocess.check_call([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared",
                           "-I", b.INCLUDE, "-I", b.CSRC, "-o", str(path / "probe.so"), str(path / "probe.cu")])
    return ctypes.CDLL(str(path / "probe.so"))


@pytest.mark.parametrize("n,status", [(1, True), (7, True), (7, False)])
def test_unfinished_instances_are_not_a_number(probe, n, status):
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    insts = torch.zeros(n * probe.inst_bytes(), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(probe.ws_bytes(), dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    partial = torch.full((n + 1,), 42.0, dtype=torch.float64, device="cuda")       # an earlier launch's
    rc = probe.probe(ptr(insts), n, ptr(ws), ptr(err) if status else None, ptr(partial),
                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    assert torch.isnan(partial[:n]).all() and partial[n].item() == 42.0
    assert err.item() == (5 if status else 0)
