"""k_tile with NaN-poisoned write buffers and guard zones against the same runs
without: nothing outside the pulled populations is read, nothing outside the
buffers written, at sizes whose tiles end past the lattice or whose halo is
wider than it."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d
from test_gpu_march import STORAGE, _workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FLAGS = lb2d.LB_DEBUG_POISON | lb2d.LB_DEBUG_GUARDS


@pytest.mark.parametrize("storage", ["fp32", "fp16_stochastic"])
@pytest.mark.parametrize("nx,ny,openings", [(9, 13, None), (61, 31, "dirichlet"), (190, 77, None), (64, 32, "poiseuille")])
def test_poisoned_tiles(nx, ny, openings, storage):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    st, kw = STORAGE[storage]
    w = _workload(nx, ny, openings)
    if nx > 100:
        w.solid[20:50, 40:120] = 1  # whole sectors without fluid
        w.rho = [np.where(w.solid, 0.0, np.where(w.rho[0] == 0, 1.0, w.rho[0]))]
    runs = []
    for flags in (0, FLAGS):
        lt = lb2d.from_workload(w, st, debug=flags, **kw)
        before = lt.launch_count()
        lt.iteration(12)
        lt.iteration(7)
        assert lt.launch_count() - before < 12  # by tiles
        runs.append([lt.populations(), *lt.velocity_f32(), *lt.fields()])
        if flags:
            assert lt.debug_check() == 0
    for x, y in zip(*runs):
        assert np.array_equal(x, y) and np.all(np.isfinite(x))
