"""A batch advanced by several calls of odd lengths against one call, bit for
bit: every call's first launch uses the work counter and the launch number
of parity 0, which the previous call's last launch has used as well."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage,kw", [("fp32", {}), ("fp16", {"h_max": 5e-3, "rounding": "stochastic"})])
def test_odd_calls_equal_one_call(storage, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    ws = synth.batch(count=5, smin=64, smax=128, step=32)
    out = []
    for calls in ([9], [1, 3, 1, 1, 3]):
        lats = [lb2d.from_workload(w, storage, **kw) for w in ws]
        b = lb2d.Batch(lats)
        for n in calls:
            b.iteration(n)
        out.append([lt.populations() for lt in lats])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
