"""How many launches short calls on small lattices take: by tiles where
these are long enough to pay, else one per iteration (launches of two or three
iterations take longer than single ones on all but the smallest)."""
import pytest

from paper_1202_0442_gb300 import lb2d
from test_gpu_march import _workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,n,launches", [(64, 32, 5, 1), (256, 256, 5, 1), (256, 256, 4, 4), (400, 400, 4, 4),
                                              (400, 400, 7, 7), (400, 400, 12, 2), (320, 320, 3, 3)])
def test_short_calls(nx, ny, n, launches):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    lt = lb2d.from_workload(_workload(nx, ny, None), thermo=1 << 30)
    lt.iteration(1)
    before = lt.launch_count()
    lt.iteration(n)
    assert lt.launch_count() - before == launches
