"""The growth step over the surface list, which each launch reads before the
kernel between it and its previous launch has ended, while that previous
launch has appended to the list and changed codes and deposits on other SMs:
a surface that grows in most steps, from fewer entries than a launch has
threads to more, against the scan of every row, bit for bit."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage,kw", [("fp32", {}), ("fp16", {"h_max": 4e-3, "rounding": "stochastic"})])
@pytest.mark.parametrize("q", [4, 9])
def test_growing_surface_list_equals_row_scan(q, storage, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    w = synth.reactive(256, 128, seed=5, ndiscs=12, rmin=4, rmax=8, q=q, kr=0.1, bmax=0.3, growth_seed=3,
                       inlet="pressure")
    whole = lb2d.from_workload(w, storage, **kw)
    one = lb2d.from_workload(w, storage, slab=(1, 0), **kw)
    for n in [1] * 40 + [25] * 4:
        whole.iteration(n)
        one.iteration(n)
        assert np.array_equal(whole.flips(), np.sort(one.flips()))
    assert np.array_equal(whole.mask(), one.mask())
    assert np.array_equal(whole.populations(1), one.populations(1))
    for a, b in zip(whole.solute_state(), one.solute_state()):
        assert np.array_equal(a, b)
    t = whole.get_thermo()
    assert t == one.get_thermo()
    assert t["flips"] > 300
