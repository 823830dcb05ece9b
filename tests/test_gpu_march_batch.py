"""The batched pairs of iterations (k_march_batch) against the batched single
ones (k_batch, calls of one iteration), bit for bit, in every storage form: a
batch large enough for the pairs in each of them, with lattices of one strip,
odd sides, fewer rows than a segment and either form of the relaxation."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d
from test_gpu_march import STORAGE, _workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(64, 512), (333, 190), (512, 480), (61, 31), (96, 5), (1, 1), (301, 299), (512, 351)]
TAUS = [0.6, 1.5, 0.8, 1.0, 0.9, 0.7, 1.2, 0.55]


@pytest.mark.parametrize("storage", list(STORAGE))
def test_large_batch_by_pairs_equals_single_iterations(storage):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    st, kw = STORAGE[storage]
    assert sum(nx * ny for nx, ny in SIZES) > 600000
    out, launches = [], []
    for calls in ([11, 24], [1] * 35):
        lats = []
        for (nx, ny), tau in zip(SIZES, TAUS):
            w = _workload(nx, ny, None)
            w.tau = (tau,)
            lats.append(lb2d.from_workload(w, st, thermo=1 << 30, **kw))
        b = lb2d.Batch(lats)
        for n in calls:
            b.iteration(n)
        launches.append(b.launch_count())
        out.append([(lt.populations(), lt.current_buffer()) for lt in lats])
    # 11: 4 pairs and 3 singles; 24: a graph of 10 and 2 pairs
    assert launches[0] < 25 and launches[1] == 35
    for (x, i), (y, j) in zip(*out):
        assert i == j and np.array_equal(x, y) and np.all(np.isfinite(x))
