"""Which launches lbm_step and lbm_batch_step make, with a fake CUDA runtime (no GPU)."""
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
