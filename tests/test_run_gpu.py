"""A run of steps in one launch (what lbm_step does by default) gives the state of the same steps
launched one by one with the one-tile kernel, bit for bit, ghost frame included.  The cases are the
forms that the order of a run's tiles distinguishes: walls and periodic y, a last tile row of one cell
row next to the first around the periodic edge (which reaches two tile rows), grids of one tile and of
one tile row, fixed and claimed tile positions, and several levels in flight (FP32 grids beyond L2)."""
import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STORAGES = ("fp32", "fp16", "bf16", "fp16_fg", "bf16_fg")


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lbm.load()
    return torch


def workload(flow, nx, ny):
    if flow == "walls":
        p, f = W.shear_drop(nx, ny, R=0.2 * min(nx, ny))
    elif flow == "periodic":
        p, f = W.stationary_drop(nx, ny, R=0.3 * min(nx, ny))
    elif flow == "prescribed":
        p, f = W.convected_drop(nx, ny, R=0.3 * min(nx, ny))
        return p, f
    else:  # density ratio 10 with gravity, walls or periodic y
        p, _ = W.rising_bubble(8.0)
        p = dict(p, nx=nx, ny=ny, walls=flow == "ratio")
        _, f = W.stationary_drop(nx, ny, R=0.3 * min(nx, ny))
    return p, W.perturbed(p, f, seed=nx + ny)


def states(torch, p, f, parts, kernel=None):
    g = lbm.Lattice(p)
    if kernel:
        g.kernel = kernel
    g.init(**f)
    for n in parts:
        g.step(n)
    torch.cuda.synchronize()
    s, ok, steps = g.state(), g.status, g.steps
    g.close()
    return s, ok, steps


def check(torch, p, f, parts):
    a = states(torch, p, f, parts)
    assert a[1] == lbm.LBM_OK and a[2] == sum(parts)
    assert a == states(torch, p, f, [sum(parts)], "tile")


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("flow,nx,ny", [
    ("walls", 33, 9), ("walls", 70, 8), ("walls", 20, 6), ("walls", 45, 25),
    ("periodic", 64, 33), ("periodic", 45, 17), ("periodic", 40, 9), ("periodic", 31, 5), ("periodic", 96, 40),
    ("prescribed", 45, 41), ("ratio", 50, 33), ("ratio_periodic", 37, 25)])
def test_small_grids(torch, storage, flow, nx, ny):
    p, f = workload(flow, nx, ny)
    check(torch, dict(p, storage=storage), f, [8, 13])


@pytest.mark.parametrize("flow,nx,ny", [("walls", 2, 2), ("periodic", 2, 2), ("periodic", 3, 2), ("walls", 3, 9)])
def test_smallest_grids(torch, flow, nx, ny):
    p, f = workload(flow, nx, ny)
    check(torch, dict(p, n_eps=1e-4), f, [40])


@pytest.mark.parametrize("storage,flow,nx,ny", [
    # fixed positions, several tiles per SM
    ("fp32", "walls", 500, 300), ("fp16", "periodic", 517, 353), ("bf16_fg", "ratio", 500, 405),
    # claimed positions
    ("fp16", "walls", 1300, 401), ("fp32", "periodic", 1026, 513), ("fp16_fg", "prescribed", 1100, 600),
    ("bf16", "ratio_periodic", 1003, 505),
    # several levels in flight
    ("fp32", "walls", 2048, 1024), ("fp32", "periodic", 1505, 1001), ("fp32", "ratio", 1024, 2047)])
def test_large_grids(torch, storage, flow, nx, ny):
    p, f = workload(flow, nx, ny)
    check(torch, dict(p, storage=storage), f, [11, 8])


def test_short_runs_and_single_steps_mix(torch):
    p, f = workload("walls", 200, 120)
    check(torch, p, f, [1, 9, 2, 8, 1, 16])


def test_run_in_a_captured_graph(torch):
    """lbm_step in a stream capture records the run; the counters are reset inside it, so replays repeat."""
    for nx, ny in ((200, 120), (1300, 400)):
        p, f = workload("walls", nx, ny)
        stream = torch.cuda.Stream()
        g = lbm.Lattice(p, stream=stream)
        g.init(**f)
        g.step(2)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.step(10)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        m = g.moments()
        g.close()
        ref = lbm.Lattice(p)
        ref.kernel = "tile"
        ref.init(**f)
        ref.step(22)
        r = ref.moments()
        ref.close()
        for k in m:
            assert (m[k] == r[k]).all(), k


def test_two_lattices_on_two_streams(torch):
    p, f = workload("walls", 300, 200)
    q, h = workload("periodic", 1100, 500)
    lats = []
    for pp, ff in ((p, f), (q, h), (p, f)):
        g = lbm.Lattice(pp, stream=torch.cuda.Stream())
        g.init(**ff)
        lats.append(g)
    for _ in range(3):
        for g in lats:
            g.step(20)
    torch.cuda.synchronize()
    got = [g.state() for g in lats]
    for g in lats:
        assert g.status == lbm.LBM_OK
        g.close()
    assert got[0] == got[2] == states(torch, p, f, [60], "tile")[0]
    assert got[1] == states(torch, q, h, [60], "tile")[0]
