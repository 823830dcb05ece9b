"""k_march and its batched form with NaN-poisoned write buffers and guard
zones against the same runs without: nothing outside the pulled populations
is read, nothing outside the buffers written."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d
from test_gpu_march import STORAGE, _workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FLAGS = lb2d.LB_DEBUG_POISON | lb2d.LB_DEBUG_GUARDS


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    yield


@pytest.mark.parametrize("storage", ["fp32", "fp16_stochastic"])
@pytest.mark.parametrize("nx,ny,openings", [(649, 501, "dirichlet"), (1024, 320, None)])
def test_poisoned_march(nx, ny, openings, storage):
    st, kw = STORAGE[storage]
    w = _workload(nx, ny, openings)
    w.solid[40:90, 100:300] = 1  # whole sectors without fluid
    w.rho = [np.where(w.solid, 0.0, np.where(w.rho[0] == 0, 1.0, w.rho[0]))]
    runs = []
    for flags in (0, FLAGS):
        lt = lb2d.from_workload(w, st, debug=flags, **kw)
        lt.iteration(10)
        lt.iteration(8)
        runs.append([lt.populations(), *lt.velocity_f32(), *lt.fields()])
        if flags:
            assert lt.debug_check() == 0
    for x, y in zip(*runs):
        assert np.array_equal(x, y) and np.all(np.isfinite(x))


def test_poisoned_march_batch():
    runs = []
    for flags in (0, FLAGS):
        lats = [lb2d.from_workload(_workload(nx, ny, None), debug=flags, thermo=1 << 30)
                for nx, ny in [(512, 480), (333, 190), (417, 512)]]
        b = lb2d.Batch(lats)
        b.iteration(9)
        runs.append([lt.populations() for lt in lats])
        if flags:
            assert all(lt.debug_check() == 0 for lt in lats)
        del b
    for x, y in zip(*runs):
        assert np.array_equal(x, y) and np.all(np.isfinite(x))
