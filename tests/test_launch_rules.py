"""Which launches lbm_step and lbm_batch_step make, with a fake CUDA runtime (no GPU)."""
import ctypes as C

import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

import fake_cuda


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return fake_cuda.Fake(str(tmp_path_factory.mktemp("fake")))


@pytest.fixture
def lib(library):
    library.reset()
    return library


def params(nx, ny, storage="fp32", **kw):
    return dict(W.base_params(nx, ny, **kw), storage=storage)


def test_few_steps_are_single_launches(lib):
    h = lib.lattice(params(128, 128))
    lib.ok(lib.step(h, 7))
    assert [r["kind"] for r in lib.launches()] == ["s"] * 7


def test_a_refused_cooperative_launch_claims_its_positions(lib):
    """A stream confined to few SMs refuses a launch whose CTAs must all be resident (error 720)."""
    h = lib.lattice(params(128, 128))
    lib.fail("r", 0, 720)
    lib.ok(lib.step(h, 20))
    assert [(r["kind"], r["status"], r["cooperative"], r["nsteps"], r["steps"]) for r in lib.launches()] == [
        ("r", 720, 1, 20, 0), ("r", 0, 0, 20, 0)]
    assert lib.steps(h) == 20


@pytest.mark.parametrize("code", [1, 700])
def test_other_launch_errors_are_reported(lib, code):
    h = lib.lattice(params(128, 128))
    lib.fail("r", 0, code)
    assert lib.step(h, 20) == lbm.LBM_ECUDA
    assert len(lib.launches()) == 1 and lib.steps(h) == 0


def test_a_failed_batch_run_leaves_every_member_with_the_steps_of_its_state(lib):
    """A member that runs alone, two groups of cohorts; the launch that fails, and what a retry starts from."""
    big, small, half = params(1100, 1024), params(300, 200), params(200, 200, "fp16")
    for at, steps in ((0, [30, 0, 0, 0]), (1, [30, 30, 30, 0])):
        lib.reset()
        hs = [lib.lattice(p) for p in (big, small, small, half)]
        b = lib.batch(hs)
        lib.fail("R", at, 700)
        assert lib.batch_step(b, 30) == lbm.LBM_ECUDA
        assert [lib.steps(h) for h in hs] == steps
        lib.reset()
        lib.ok(lib.batch_step(b, 30))
        assert [lib.steps(h) for h in hs] == [s + 30 for s in steps]
        assert [r["steps"] for r in lib.launches()] == [steps[0], steps[1], steps[3]]


def test_a_batch_run_that_fails_after_others_counts_those(lib):
    hs = [lib.lattice(params(512, 700)) for _ in range(12)]
    b = lib.batch(hs)
    lib.fail("R", 1, 700)
    assert lib.batch_step(b, 5000) == lbm.LBM_ECUDA
    done = lib.launches()[0]["nsteps"]
    assert 0 < done < 5000 and [lib.steps(h) for h in hs] == [done] * 12


@pytest.mark.parametrize("nx,ny,storage,n", [(8, 8, "fp16", 10000), (128, 128, "fp32", 20000), (2048, 1024, "fp32", 3000),
                                             (2048, 1024, "fp16", 1000), (4096, 4096, "fp32", 200), (8192, 16000, "fp16", 50)])
def test_a_run_ends_within_some_milliseconds(lib, nx, ny, storage, n):
    """A tile's update takes some 8 ns at most and a step 4 us at least: no launch beyond 40 ms."""
    h = lib.lattice(params(nx, ny, storage))
    lib.ok(lib.step(h, n))
    done = lib.launches()
    assert any(r["kind"] == "r" for r in done)
    assert sum(r["nsteps"] for r in done) == n == lib.steps(h)
    assert all(max(r["nsteps"] * r["tiles"] * 8e-9, r["nsteps"] * 4e-6) < 0.04 for r in done)


def test_a_batch_run_ends_within_some_milliseconds(lib):
    hs = [lib.lattice(params(1000, 768)) for _ in range(96)] + [lib.lattice(params(16640, 16000))]
    for h in hs[-1:]:
        lib.ok(lib.lib.lbm_set_kernel(h, lbm.LBM_KERNEL_TILE))  # joins the others instead of running alone
    for members in (hs[:8], hs):
        lib.reset()
        before = [lib.steps(h) for h in members]
        b = lib.batch(members)
        lib.ok(lib.batch_step(b, 600))
        assert [lib.steps(h) for h in members] == [s + 600 for s in before]
        assert all(max(r["nsteps"] * r["tiles"] * 8e-9, r["nsteps"] * 4e-6) < 0.04 for r in lib.launches())


@pytest.mark.parametrize("nx,ny", [(20000, 16000), (2048, 16136)])
def test_the_largest_grids_go_step_by_step(lib, nx, ny):
    """More than 2^20 tiles, or more tile rows than there are counters."""
    h = lib.lattice(params(nx, ny))
    lib.ok(lib.step(h, 20))
    assert [r["kind"] for r in lib.launches()] == ["s"] * 20


def test_a_batch_sets_a_kernel_up_once(lib):
    hs = [lib.lattice(params(64, 64)), lib.lattice(params(96, 64)), lib.lattice(params(64, 64, "fp16"))]
    b = lib.batch(hs)
    assert lib.prepared("R") == 2
    arr = (C.c_void_p * 2)(hs[0], hs[2])
    for _ in range(3):
        lib.ok(lib.lib.lbm_batch_set_schedule(b, 1, 0))
        lib.ok(lib.lib.lbm_batch_set_members(b, arr, 2))
    assert lib.prepared("R") == 2
    lib.ok(lib.lib.lbm_batch_set_members(b, (C.c_void_p * 1)(lib.lattice(params(64, 64, walls=True))), 1))
    assert lib.prepared("R") == 3


def path(lib, p, n):
    lib.reset()
    lib.ok(lib.step(lib.lattice(p), n))
    return "".join(r["kind"] for r in lib.launches())


FLOWS = {"solved": dict(walls=True), "periodic": {}, "ratio": dict(walls=True, rhoA=1.0, rhoB=0.1),
         "prescribed": dict(velocity="prescribed")}


@pytest.mark.parametrize("storage,flow,nx,ny,never", [
    ("fp32", "solved", 64, 64, True), ("fp32", "solved", 128, 128, False),      # few tiles
    ("fp32", "prescribed", 128, 128, True), ("fp32", "ratio", 64, 64, False),
    ("fp32", "prescribed", 300, 300, True), ("fp32", "prescribed", 160, 160, False),
    ("fp16", "solved", 300, 300, True), ("fp16", "solved", 128, 128, False),    # one to three tiles per SM
    ("fp32", "solved", 100000, 8, True), ("fp16", "ratio", 50000, 32, True),    # few tile rows
    ("fp16", "solved", 50000, 32, False), ("fp32", "solved", 4000, 8, False), ("fp16", "periodic", 4000, 33, False),
    ("fp16", "periodic", 120, 1600, True), ("fp16", "periodic", 250, 800, False),           # narrow
    ("bf16_fg", "ratio", 180, 1100, True), ("fp16", "solved", 120, 1600, False), ("fp16", "solved", 250, 2000, True),
    ("fp16", "solved", 280, 2000, False), ("fp32", "periodic", 120, 1600, False),
    ("fp16", "prescribed", 120, 1600, False)])
def test_grids_that_are_faster_step_by_step_take_no_runs(lib, storage, flow, nx, ny, never):
    assert path(lib, params(nx, ny, storage, **FLOWS[flow]), 64) == ("s" * 64 if never else "r")


@pytest.mark.parametrize("storage,flow,nx,ny,fewest", [
    ("fp32", "solved", 1024, 1024, 4), ("fp32", "solved", 300, 300, 8), ("fp32", "prescribed", 620, 620, 12),
    ("fp32", "prescribed", 420, 420, 16), ("fp16", "solved", 700, 600, 4), ("fp16", "ratio", 700, 600, 8),
    ("fp16", "ratio", 1024, 1024, 4), ("fp16", "solved", 64, 64, 16), ("bf16_fg", "prescribed", 64, 64, 32)])
def test_few_steps_of_a_grid_go_one_by_one(lib, storage, flow, nx, ny, fewest):
    p = params(nx, ny, storage, **FLOWS[flow])
    assert path(lib, p, fewest - 1) == "s" * (fewest - 1) and path(lib, p, fewest) == "r"


def batch_path(lib, members, n, graph_steps=0):
    b = lib.batch([lib.lattice(p) for p in members])
    lib.ok(lib.lib.lbm_batch_set_schedule(b, 1, graph_steps))
    lib.reset()
    lib.ok(lib.batch_step(b, n))
    return "".join(r["kind"] for r in lib.launches())


def test_batches_that_are_faster_step_by_step_take_no_runs(lib):
    small, flat = [params(64, 64)] * 4, [params(100000, 8), params(300, 300)]
    assert batch_path(lib, small, 15) == "b" * 15 and batch_path(lib, small, 16) == "R"
    assert "R" not in batch_path(lib, small, 48, graph_steps=16) and batch_path(lib, small, 64, graph_steps=16) == "R"
    assert batch_path(lib, flat, 64) == "b" * 64


def test_members_of_half_storage_run_alone_from_their_own_size_on(lib):
    for flow, nx, alone in (("solved", 700, True), ("prescribed", 700, False), ("ratio", 700, False),
                            ("prescribed", 850, True), ("ratio", 850, True)):
        assert batch_path(lib, [params(nx, nx, "fp16", **FLOWS[flow])] * 2, 64) == ("rr" if alone else "R")


def test_launches_are_counted(lib):
    h, n = lib.lattice(params(128, 128)), C.c_int64()
    for steps, total in ((5, 5), (20, 6), (9000, 9)):
        lib.ok(lib.step(h, steps))
        lib.ok(lib.lib.lbm_launches(h, C.byref(n)))
        assert n.value == total == len(lib.launches())
    assert lib.lib.lbm_launches(None, C.byref(n)) == lbm.LBM_EINVAL


def test_a_narrow_member_joins_the_others(lib):
    narrow = params(250, 4000, "fp16")
    assert path(lib, narrow, 64) == "s" * 64 and batch_path(lib, [narrow] * 2, 64) == "R"
