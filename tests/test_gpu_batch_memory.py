"""A batch gives back what it allocated: creating and destroying batches that
advance two iterations per launch (the largest form of their device arrays)
leaves the free device memory where it was."""
import pytest

from paper_1202_0442_gb300 import lb2d, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_destroyed_batches_leave_no_device_memory():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    lats = [lb2d.from_workload(w) for w in synth.batch(count=16, smin=192, smax=512, step=32)]
    assert sum(lt.nx * lt.ny for lt in lats) > 1000000

    def use(n):
        for _ in range(n):
            b = lb2d.Batch(lats)
            b.iteration(8, use_graph=False)
            assert b.launch_count() < 8  # by pairs
            del b
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    before = use(3)
    # 32 descriptors and some 1500 tasks of 16 bytes: 400 batches that kept
    # them would hold some 10 MB, several of the allocator's 2 MB pages
    assert use(400) == before
