"""Which lattices go by two iterations per launch, told by the launch count:
wide ones, and not the narrow ones with openings or the batches of badly
filled strips, which take longer that way."""
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
@pytest.mark.parametrize("nx,ny,pairs", [(58, 12000, False), (122, 6000, False), (180, 6000, True), (660, 660, True),
                                         (200, 20000, True)])
def test_lattice(nx, ny, pairs, storage):
    st, kw = STORAGE[storage]
    lt = lb2d.from_workload(_workload(nx, ny, "dirichlet"), st, thermo=1 << 30, **kw)
    lt.iteration(1)
    before = lt.launch_count()
    lt.iteration(8)
    assert lt.launch_count() - before == (4 if pairs else 8)


@pytest.mark.parametrize("storage", ["fp32", "fp32_precise", "fp16_stochastic"])
@pytest.mark.parametrize("count,nx,ny,pairs", [(66, 122, 122, False), (22, 100, 300, True)])
def test_batch(count, nx, ny, pairs, storage):
    st, kw = STORAGE[storage]
    w = _workload(nx, ny, None)
    b = lb2d.Batch([lb2d.from_workload(w, st, thermo=1 << 30, **kw) for _ in range(count)])
    b.iteration(8, use_graph=False)
    assert b.launch_count() == (4 if pairs else 8)
