"""lbm_reduce, whose last block adds the partial sums, against lbm_reduce_noalloc, which adds them in a
second launch: the same partial sums in the same order up to 1024 rows, so the same bits; beyond, a
block holds several rows and the order differs."""
import pytest

from paper_2408_15654_gb300 import lbm
from paper_2408_15654_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (33, 5), (300, 255), (28, 257), (40, 1024), (31, 1025)])
def test_one_launch_sum_equals_two_launches(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, f = W.stationary_drop(nx, ny, R=0.3 * min(nx, ny))
    sim = lbm.Lattice(p)
    sim.init(**W.perturbed(p, f, seed=5))
    sim.step(3)
    pitch = (nx + 10 + 31) // 32 * 32
    buf = (26 * (ny + 4) * pitch * 4 + 255) // 256 * 256
    for what in (lbm.LBM_SUM_PHI, lbm.LBM_SUM_PSI, lbm.LBM_SUM_PHI):
        got = lbm.lbm_reduce(sim.handle, what)
        two = lbm.lbm_reduce_noalloc(sim.workspace.data_ptr() + (sim.steps % 2) * buf, nx, ny, what,
                                     sim.stream.cuda_stream)
        assert got == two if ny <= 1024 else got == pytest.approx(two, rel=1e-12)
        assert got == lbm.lbm_reduce(sim.handle, what)
    sim.close()
