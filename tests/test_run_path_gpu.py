"""Runs of steps are taken where the library says so, by its count of launches, and give there the state of one
launch per step, bit for bit: the forms that the order of a run's tiles distinguishes, on grids that take runs
(FP32 storage at uniform density: from 56 or 80 tiles on), claims of eight tiles, and members of a batch alone."""
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


def workload(flow, nx, ny, storage):
    if flow == "prescribed":
        p, f = W.convected_drop(nx, ny, R=0.3 * min(nx, ny))
        return dict(p, storage=storage), f
    if flow in ("walls", "periodic"):
        p, f = (W.shear_drop if flow == "walls" else W.stationary_drop)(nx, ny, R=0.25 * min(nx, ny))
    else:  # density ratio 10 with gravity, walls or periodic y
        p, _ = W.rising_bubble(8.0)
        p = dict(p, nx=nx, ny=ny, walls=flow == "ratio")
        _, f = W.stationary_drop(nx, ny, R=0.3 * min(nx, ny))
    return dict(p, storage=storage), W.perturbed(p, f, seed=nx + ny)


def check(p, f, parts, launches):
    """`parts` calls take `launches` launches in all, and as many as steps with the one-tile kernel."""
    state = []
    for kernel, count in (("auto", launches), ("tile", sum(parts))):
        g = lbm.Lattice(p)
        g.kernel = kernel
        g.init(**f)
        for n in parts:
            g.step(n)
        assert g.status == lbm.LBM_OK and g.steps == sum(parts)
        assert g.launches == count, (kernel, g.launches)
        state.append(g.state())
        g.close()
    assert state[0] == state[1]


@pytest.mark.parametrize("flow,nx,ny", [
    ("walls", 1000, 9), ("walls", 2000, 8), ("walls", 600, 25), ("walls", 333, 57), ("walls", 70, 600),
    ("periodic", 500, 33), ("periodic", 600, 25), ("periodic", 900, 17), ("periodic", 1000, 9), ("periodic", 2000, 5),
    ("periodic", 500, 40), ("periodic", 33, 241), ("prescribed", 700, 41), ("prescribed", 900, 24)])
def test_fp32_at_uniform_density(torch, flow, nx, ny):
    p, f = workload(flow, nx, ny, "fp32")
    check(p, f, [12, 13], 2)


@pytest.mark.parametrize("storage", ["fp16", "bf16", "fp16_fg", "bf16_fg"])
@pytest.mark.parametrize("flow,nx,ny", [
    ("walls", 33, 9), ("walls", 70, 8), ("walls", 20, 6), ("walls", 45, 25), ("periodic", 64, 33), ("periodic", 45, 17),
    ("periodic", 40, 9), ("periodic", 31, 5), ("periodic", 96, 40), ("prescribed", 45, 41), ("ratio", 50, 33),
    ("ratio_periodic", 37, 25)])
def test_few_tiles_of_half_storage(torch, storage, flow, nx, ny):
    p, f = workload(flow, nx, ny, storage)
    check(dict(p, n_eps=1e-4), f, [33, 32], 2)


@pytest.mark.parametrize("flow,nx,ny", [("ratio", 50, 33), ("ratio_periodic", 37, 25), ("ratio", 33, 9), ("ratio", 2, 2),
                                        ("ratio_periodic", 3, 9)])
def test_fp32_with_a_density_ratio(torch, flow, nx, ny):
    p, f = workload(flow, nx, ny, "fp32")
    check(dict(p, n_eps=1e-4), f, [9, 8], 2)


@pytest.mark.parametrize("flow,nx,ny", [("walls", 2048, 1024), ("periodic", 2048, 1000), ("periodic", 2048, 1001)])
def test_claims_of_the_largest_half_storage_grids(torch, flow, nx, ny):
    """Eight tiles a claim; four with a reach of two tile rows."""
    p, f = workload(flow, nx, ny, "fp16")
    check(p, f, [11, 8], 2)


@pytest.mark.parametrize("storage,nx,ny", [("fp16", 300, 300), ("fp32", 64, 64), ("fp32", 100000, 8)])
def test_grids_that_take_no_runs(torch, storage, nx, ny):
    p, f = workload("walls", nx, ny, storage)
    check(p, f, [40], 40)


def test_members_alone_and_together(torch):
    """A member with a chosen kernel joins the others; the large ones advance by their own runs."""
    stream = torch.cuda.Stream()
    sizes = [(1100, 1024), (1000, 1024), (300, 200), (1000, 1024)]
    lats = []
    for k, (nx, ny) in enumerate(sizes):
        p, f = workload("walls", nx, ny, "fp32")
        g = lbm.Lattice(dict(p, E0=0.1 + 0.01 * k), stream=stream)
        g.init(**f)
        lats.append(g)
    lats[0].kernel = "tile"
    b = lbm.Batch(lats, stream)
    b.step(20)
    assert [g.launches for g in lats] == [0, 1, 0, 1]
    assert b.launches == 2 + 2  # two members alone; the run of the others and the reset of its counters
    b.step(3)
    assert [g.launches for g in lats] == [0, 1, 0, 1]
    b.close()
    for g in lats:
        assert g.status == lbm.LBM_OK and g.steps == 23
        g.close()
