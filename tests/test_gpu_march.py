"""Two iterations per launch (k_march) against one at a time
(lb_set_kernel "streaming"), bit for bit: populations, node fields, thermo
records and the current buffer, at the widths and heights where its strips
and segments end (one strip, odd widths whose last pair wraps, a lane's pair
across the edge, a last strip of one column, a single row), with openings on the x walls, for every
storage form.  An iteration count that is not a multiple of four leaves
single iterations between the pairs and the record."""
import numpy as np
import pytest

from paper_1202_0442_gb300 import lb2d, synth

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


STORAGE = {
    "fp32": ("fp32", {}),
    "fp32_precise": ("fp32", {"precise": True}),
    "fp16_stochastic": ("fp16", {"h_max": 2e-2, "rounding": "stochastic"}),
    "fp16_nearest": ("fp16", {"h_max": 2e-2}),
    "bf16_stochastic": ("bf16", {"rounding": "stochastic"}),
}


def _workload(nx, ny, openings):
    rng = np.random.default_rng(nx * 7 + ny)
    m = (rng.random((ny, nx)) < 0.2).astype(np.uint8)
    ops = []
    if openings:
        m[:, :2] = m[:, -2:] = 0
        first = {"dirichlet": ("dirichlet", 0.0, 1.001), "poiseuille": ("poiseuille", 0.01, 1.0)}[openings]
        ops = [synth.Opening("xlo", 1, ny - 3, "inlet", [first]),
               synth.Opening("xhi", 2, ny - 1, "outlet",
                             [("dirichlet", 0.0, 1.0) if openings == "dirichlet" else ("uniform", 0.004, 1.0)])]
    u = lambda: 1e-3 * rng.standard_normal((ny, nx))
    return synth.Workload(name="march", nx=nx, ny=ny, solid=m,
                          rho=[np.where(m, 0.0, 1.0 + 1e-3 * rng.random((ny, nx)))], ux=u(), uy=u(), tau=(0.8,),
                          aveforce=((1e-5, 2e-6),), aveacceleration=((3e-6, 0.0),), openings=ops)


@pytest.mark.parametrize("storage", list(STORAGE))
@pytest.mark.parametrize("openings", [None, "dirichlet", "poiseuille"])
@pytest.mark.parametrize("nx,ny", [(39, 8300), (121, 2700), (649, 501), (1025, 313), (1741, 190), (3601, 90), (320001, 1)])
def test_march_equals_single_iterations(nx, ny, openings, storage):
    if openings and ny < 8:
        pytest.skip("the openings' spans need a few rows")
    st, kw = STORAGE[storage]
    w = _workload(nx, ny, openings)
    a = lb2d.from_workload(w, st, kernel="streaming", **kw)
    b = lb2d.from_workload(w, st, **kw)
    for n in (11, 8):
        for lt in (a, b):
            lt.iteration(n)
        assert a.current_buffer() == b.current_buffer()
        assert a.get_thermo() == b.get_thermo()
        assert np.array_equal(a.populations(), b.populations())
        for x, y in zip(a.velocity_f32(), b.velocity_f32()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.fields()[3], b.fields()[3])
    assert b.launch_count() < a.launch_count() - 6


@pytest.mark.parametrize("storage", list(STORAGE))
def test_batch_by_pairs_equals_single_iterations(storage):
    """The batched launch's pairs of iterations against its single ones (calls
    of one iteration), bit for bit, over lattices of uneven sizes (one strip,
    odd sides, fewer rows than a segment, either form of the relaxation)."""
    st, kw = STORAGE[storage]
    sizes = [(64, 512), (333, 190), (512, 480), (61, 31), (96, 5), (1, 1), (301, 299)]
    taus = [0.6, 1.5, 0.8, 1.0, 0.9, 0.7, 1.2]
    out = []
    for calls in ([11, 24], [1] * 35):
        lats = []
        for k, ((nx, ny), tau) in enumerate(zip(sizes, taus)):
            w = _workload(nx, ny, None)
            w.tau = (tau,)
            lats.append(lb2d.from_workload(w, st, thermo=1 << 30, **kw))
        b = lb2d.Batch(lats)
        for n in calls:
            b.iteration(n)
        out.append([(lt.populations(), lt.current_buffer()) for lt in lats])
        launches = b.launch_count()
    assert launches == 35
    for (x, i), (y, j) in zip(*out):
        assert i == j and np.array_equal(x, y)
