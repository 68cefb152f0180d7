"""Streams whose work runs on a part of the GPU only (a green context): runs of steps, whose launches may
need all their CTAs resident at once, give the same state there as one launch per step."""
import ctypes as C

import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RESOURCE_BYTES, SM_COUNT_OFFSET, TYPE_SM = 144, 96, 1  # CUdevResource of cuda.h


@pytest.fixture(scope="module")
def confined():
    """A stream on 16 of the SMs."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lbm.load()
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    dev, desc, ctx, stream = C.c_int(), C.c_void_p(), C.c_void_p(), C.c_void_p()
    every, part, rest = (C.create_string_buffer(RESOURCE_BYTES) for _ in range(3))
    groups = C.c_uint(1)
    for name, *args in (("cuDeviceGet", C.byref(dev), 0), ("cuDeviceGetDevResource", dev, every, TYPE_SM),
                        ("cuDevSmResourceSplitByCount", part, C.byref(groups), every, rest, 0, 16),
                        ("cuDevResourceGenerateDesc", C.byref(desc), part, 1),
                        ("cuGreenCtxCreate", C.byref(ctx), desc, dev, 1)):
        if getattr(cu, name)(*args):
            pytest.skip(f"no green contexts: {name}")
    assert 0 < C.c_uint.from_buffer(part, SM_COUNT_OFFSET).value < 64
    assert cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0) == 0
    yield torch, torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("storage,nx,ny", [("fp32", 128, 128), ("fp16", 500, 600), ("fp32", 700, 512), ("fp16", 1300, 401),
                                           ("fp32", 1505, 1001)])
def test_runs_on_a_part_of_the_gpu(confined, storage, nx, ny):
    torch, stream = confined
    p, f = W.shear_drop(nx, ny, R=0.2 * ny)
    p, f = dict(p, storage=storage), W.perturbed(p, f, seed=nx)
    state = []
    for kernel in ("auto", "tile"):
        g = lbm.Lattice(p, stream=stream)
        g.kernel = kernel
        g.init(**f)
        g.step(12)
        g.step(9)
        assert g.status == lbm.LBM_OK and g.steps == 21
        state.append(g.state())
        g.close()
    assert state[0] == state[1]
