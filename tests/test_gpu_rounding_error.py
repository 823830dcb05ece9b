"""How far FP32 storage's rounding carries a pressure-driven channel flow from
the FP64 oracle in 200 iterations (relative 2-norm of the deviations from the
rest state).  The bound is what the collision's plain FP32 form (u from a
rounded reciprocal, the quadratic terms from rho and u, the diagonal
antisymmetric parts rounded once) gives on this flow in an emulation with
numpy, so that no rearranged form of the equilibrium may do worse; one whose
antisymmetric parts came from fused products of (mx + my) gives 2.1e-7."""
import numpy as np
import pytest

from oracle.drive import oracle_from_workload
from paper_1202_0442_gb300 import lb2d, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STEPS = 200
PLAIN = 1.8e-7


def workload():
    w = synth.reactive(1024, 512, seed=3, ndiscs=40, inlet="pressure")
    w.solute_q, w.reaction, w.C = 0, None, None
    for op in w.openings:
        op.solute = None
    x, y = np.arange(w.nx) * (2 * np.pi / w.nx), np.arange(w.ny) * (2 * np.pi / w.ny)
    w.ux = 1e-3 * np.outer(np.sin(y + 0.3), np.cos(2 * x + 1.1))
    w.uy = 1e-3 * np.outer(np.cos(2 * y + 0.7), np.sin(x + 2.0))
    return w


@pytest.mark.parametrize("kernel", ["auto", "streaming"])
def test_rounding_error_of_a_channel_flow(kernel):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    w = workload()
    lt = lb2d.from_workload(w, kernel=kernel)
    o = oracle_from_workload(w)
    lt.iteration(STEPS)
    o.step(STEPS)
    fluid = w.solid == 0
    rest = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None]
    h, ref = (f.reshape(9, w.ny, w.nx)[:, fluid] - rest for f in (lt.populations(), o.f()))
    assert np.linalg.norm(h - ref) < PLAIN * np.linalg.norm(ref)


@pytest.mark.parametrize("kernel", ["auto", "streaming"])
def test_exact_momentum_in_a_slow_porous_flow(kernel):
    """Exact momentum pairs on a slow force-driven porous lattice, 5000
    iterations: the velocity's error (2-norm over the fluid nodes, of the
    largest velocity) is 7.8e-8 for the plain form in the emulation, 8.7e-8
    with unrounded antisymmetric parts and 1.6e-7 with rounded ones."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1202_0442_gb300 import build
    build.build()
    w = synth.batch(count=110)[109]
    lt = lb2d.from_workload(w, kernel=kernel, precise=True)
    o = oracle_from_workload(w)
    lt.iteration(5000)
    o.step(5000)
    fluid = w.solid == 0
    u = [a.astype(np.float64) for a in lt.velocity_f32()[1:]]
    ref = o.velocity()
    err = np.sqrt(np.mean((u[0] - ref[0])[fluid] ** 2 + (u[1] - ref[1])[fluid] ** 2) * fluid.mean())
    assert err < 1.2e-7 * max(np.max(np.abs(b[fluid])) for b in ref)
