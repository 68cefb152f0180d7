"""The waits inside a run of steps end: tiles that wait for a tile that nobody updates give up within seconds,
without a fault, LBM_ETIMEOUT tells so for every lattice of the launch, and lattices step as before afterwards."""
import time

import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lbm.load()
    return torch


def workload(nx, ny, storage):
    p, f = W.shear_drop(nx, ny, R=0.2 * ny)
    return dict(p, storage=storage), W.perturbed(p, f, seed=nx)


def steps_as_one_by_one(p, f):
    state = []
    for kernel in ("auto", "tile"):
        g = lbm.Lattice(p)
        g.kernel = kernel
        g.init(**f)
        g.step(16)
        assert g.status == lbm.LBM_OK
        state.append(g.state())
        g.close()
    assert state[0] == state[1]


@pytest.mark.parametrize("storage,nx,ny", [("fp32", 128, 128), ("fp32", 700, 512), ("fp16", 128, 128), ("fp16", 1100, 600),
                                           ("bf16_fg", 500, 600), ("fp32", 2048, 1024)])
def test_a_stalled_run_gives_up(torch, storage, nx, ny):
    p, f = workload(nx, ny, storage)
    g = lbm.Lattice(p)
    g.init(**f)
    lbm.lbm_selftest_stall(g.handle, True)
    t0 = time.time()
    g.step(16)
    torch.cuda.synchronize()
    assert time.time() - t0 < 15.0
    assert g.status == lbm.LBM_ETIMEOUT
    lbm.lbm_selftest_stall(g.handle, False)
    g.init(**f)                            # clears the status and the state
    g.step(16)
    assert g.status == lbm.LBM_OK
    g.close()
    steps_as_one_by_one(p, f)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_a_stalled_member_ends_the_run_of_its_batch(torch, storage):
    stream = torch.cuda.Stream()
    work = [workload(nx, ny, storage) for nx, ny in ((256, 128), (300, 200), (64, 32))]
    lats = [lbm.Lattice(p, stream=stream) for p, _ in work]
    for g, (_, f) in zip(lats, work):
        g.init(**f)
    b = lbm.Batch(lats, stream)
    lbm.lbm_selftest_stall(lats[1].handle, True)
    t0 = time.time()
    b.step(16)
    torch.cuda.synchronize()
    assert time.time() - t0 < 15.0
    assert [g.status for g in lats] == [lbm.LBM_ETIMEOUT] * 3
    lbm.lbm_selftest_stall(lats[1].handle, False)
    for g, (_, f) in zip(lats, work):
        g.init(**f)
    b.step(16)
    for g, (p, f) in zip(lats, work):
        alone = lbm.Lattice(p)
        alone.kernel = "tile"
        alone.init(**f)
        alone.step(16)
        assert g.status == lbm.LBM_OK and g.state() == alone.state()
        alone.close()
    b.close()
    for g in lats:
        g.close()
