"""Several iterations of a small lattice per launch (k_tile) against one at a
time (lb_set_kernel "streaming"), bit for bit: populations, node fields,
thermo records and the current buffer, from a single node to the largest
lattice it serves, odd sides (tiles that end past the lattice, pairs of rows
past a tile), halos wider than the lattice, openings on the x walls, every
storage form; calls whose iterations do not divide evenly."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d
from test_gpu_march import STORAGE, _workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    yield


@pytest.mark.parametrize("storage", list(STORAGE))
@pytest.mark.parametrize("openings", [None, "dirichlet", "poiseuille"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (9, 13), (64, 32), (61, 31), (31, 700), (333, 190), (400, 400)])
def test_tiles_equal_single_iterations(nx, ny, openings, storage):
    if openings and min(nx, ny) < 8:
        pytest.skip("the openings' spans need a few rows")
    st, kw = STORAGE[storage]
    w = _workload(nx, ny, openings)
    if nx * ny < 16:
        w.solid[:] = 0
        w.rho = [np.where(w.rho[0] == 0, 1.0, w.rho[0])]
    a = lb2d.from_workload(w, st, kernel="streaming", **kw)
    b = lb2d.from_workload(w, st, **kw)
    for n in (11, 3, 4, 40):
        for lt in (a, b):
            lt.iteration(n)
        assert a.current_buffer() == b.current_buffer()
        assert a.get_thermo() == b.get_thermo()
        assert np.array_equal(a.populations(), b.populations())
        for x, y in zip(a.velocity_f32(), b.velocity_f32()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.fields()[3], b.fields()[3])
    assert b.launch_count() < a.launch_count() - 20
