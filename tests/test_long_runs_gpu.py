"""More steps than one launch of a run takes (4096, or 2^22 updates of a tile): the state of the same steps
launched one by one, bit for bit, also where a launch ends after an odd number of steps."""
import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def state(p, f, n, kernel):
    g = lbm.Lattice(p)
    g.kernel = kernel
    g.init(**f)
    g.step(n)
    s, ok, steps = g.state(), g.status, g.steps
    g.close()
    assert ok == lbm.LBM_OK and steps == n
    return s


@pytest.mark.parametrize("storage,nx,ny,n", [("fp16", 64, 64, 4096 + 77), ("fp32", 128, 128, 2 * 4096 + 9),
                                             ("fp32", 2048, 1000, 524 + 21), ("bf16_fg", 1531, 787, 882 + 30)])
def test_one_lattice(storage, nx, ny, n):
    pytest.importorskip("torch")
    p, f = W.shear_drop(nx, ny, R=0.2 * ny)
    p, f = dict(p, storage=storage, n_eps=1e-4), W.perturbed(p, f, seed=nx)
    assert state(p, f, n, "auto") == state(p, f, n, "tile")


def test_a_batch():
    """12 lattices of 1408 tiles: 248 steps a launch."""
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    p, f = W.shear_drop(512, 700, R=100)
    f = W.perturbed(p, f, seed=3)
    ps = [dict(p, E0=0.1 + 0.01 * k, n_eps=1e-4) for k in range(12)]
    lats = [lbm.Lattice(q, stream=stream) for q in ps]
    for g in lats:
        g.init(**f)
    b = lbm.Batch(lats, stream)
    b.step(263)
    for k in (0, 7, 11):
        assert lats[k].status == lbm.LBM_OK
        assert lats[k].state() == state(ps[k], f, 263, "tile")
    b.close()
    for g in lats:
        g.close()
