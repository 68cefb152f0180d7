"""A run of many steps of a batch's lattices in one launch (what lbm_batch_step does from eight steps on)
gives every member the state of the same steps launched one by one, bit for bit.  The cases are the forms
that its order of tiles distinguishes: several cohorts and more members than one launch holds, walls
and periodic y with last tile rows of one cell row (which reach two tile rows), members that run alone,
and more steps than one launch takes."""
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


def lattice(stream, flow, nx, ny, storage, k):
    if flow == "ratio":
        p, _ = W.rising_bubble(8.0)
        p = dict(p, nx=nx, ny=ny)
        _, f = W.stationary_drop(nx, ny, R=0.3 * min(nx, ny))
    elif flow == "prescribed":
        p, f = W.convected_drop(nx, ny, R=0.3 * min(nx, ny))
    else:
        make = W.shear_drop if flow == "walls" else W.stationary_drop
        p, f = make(nx, ny, R=0.25 * min(nx, ny))
    p = dict(p, storage=storage, E0=0.1 + 0.001 * k)
    g = lbm.Lattice(p, stream=stream)
    g.init(**(f if flow == "prescribed" else W.perturbed(p, f, seed=k)))
    return g


def check(torch, sizes, steps, checked, flow, storage, chosen=()):
    """Batch the lattices for calls of `steps` and 8 steps; the checked members against one-tile launches.
    The chosen members have the one-tile kernel set for their own steps."""
    stream = torch.cuda.Stream()
    lats = [lattice(stream, flow, nx, ny, storage, k) for k, (nx, ny) in enumerate(sizes)]
    for k in chosen:
        lats[k].kernel = "tile"
    b = lbm.Batch(lats, stream)
    b.step(steps)
    b.step(8)
    torch.cuda.synchronize()
    for k in checked:
        g = lattice(stream, flow, *sizes[k], storage, k)
        g.kernel = "tile"
        g.step(steps + 8)
        assert lats[k].status == g.status and lats[k].steps == steps + 8
        assert lats[k].state() == g.state(), f"member {k}"
        g.close()
    b.close()
    for g in lats:
        g.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16_fg"])
@pytest.mark.parametrize("flow", ["walls", "periodic", "ratio", "prescribed"])
def test_cohorts_and_member_chunks(torch, flow, storage):
    """104 members (a launch holds 96), several cohorts; ny = 121, 33, 17 leave a row of one cell."""
    sizes = [(256, 128), (250, 121), (97, 33), (64, 17)] * 26
    check(torch, sizes, 9, range(0, 104, 7), flow, storage)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_alone_together_and_few(torch, storage):
    check(torch, [(1100, 1024), (300, 200), (40, 9)], 9, range(3), "walls", storage)
    check(torch, [(40, 24), (2, 2)], 12, range(2), "periodic", storage)


def test_large_member_with_a_chosen_kernel(torch):
    """It joins the others; a smaller member after it still runs alone."""
    check(torch, [(1100, 1024), (1000, 1024), (300, 200)], 9, range(3), "walls", "fp32", chosen=(0,))


def test_more_steps_than_one_launch(torch):
    """12 members of 1408 tiles: a launch takes 64 steps."""
    check(torch, [(512, 700)] * 12, 66, (0, 5, 11), "walls", "fp32")
