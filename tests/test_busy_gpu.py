"""Runs of steps on a GPU that another kernel keeps busy: the CTAs that find no room wait for longer than the
waits inside a run last (a second), and the state is that of one launch per step all the same."""
import ctypes as C
import os
import subprocess
import time

import pytest

from paper_2408_15654_gb300 import build as _build
from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# holds its SMs (200 KB of shared memory each) for `ns`, and at most for some 10^7 sleeps
HOLD = r"""
#include <cuda_runtime.h>
__global__ void hold(unsigned long long ns) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (unsigned i = 0; i < 10000000u; ++i) {
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 > ns) break;
        __nanosleep(500);
    }
}
extern "C" int start_hold(int ctas, unsigned long long ns, void* stream) {
    cudaError_t e = cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess) {
        hold<<<ctas, 32, 200 * 1024, static_cast<cudaStream_t>(stream)>>>(ns);
        e = cudaGetLastError();
    }
    return e;
}
"""


@pytest.fixture(scope="module")
def start_hold(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("hold")
    (d / "hold.cu").write_text(HOLD)
    path = os.path.join(d, "hold.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", path, str(d / "hold.cu")], check=True)
    return C.CDLL(path).start_hold


@pytest.mark.parametrize("storage,nx,ny,sms", [("fp32", 608, 512, 100), ("fp16", 128, 128, 140), ("fp16", 1100, 600, 100)])
def test_a_run_waits_for_its_sms(start_hold, storage, nx, ny, sms):
    import torch

    p, f = W.shear_drop(nx, ny, R=0.2 * ny)
    p, f = dict(p, storage=storage), W.perturbed(p, f, seed=nx)
    other, stream = torch.cuda.Stream(), torch.cuda.Stream()
    state = []
    for kernel in ("auto", "tile"):
        g = lbm.Lattice(p, stream=stream)
        g.kernel = kernel
        g.init(**f)
        g.step(32)
        torch.cuda.synchronize()
        if kernel == "auto":
            assert start_hold(sms, C.c_ulonglong(1_500_000_000), C.c_void_p(other.cuda_stream)) == 0
            time.sleep(0.01)
        g.step(64)
        torch.cuda.synchronize()
        assert g.status == lbm.LBM_OK and g.steps == 96
        state.append(g.state())
        g.close()
    assert state[0] == state[1]
