"""Double storage: the integer moment sums and the corrected Landau frame against the oracle, at the
scales and velocities where their grids and branches change."""
import numpy as np
import pytest

import oracle
from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, RLBError  # noqa: E402
from paper_1301_3423_gb300.rlb import RLB_ENONCONV  # noqa: E402


def pair(lat, order, n, T, u, steps):
    shape = n.shape
    o = oracle.OracleRLB(lat, shape[2], shape[1], shape[0], eta_over_s=0.1)
    o.init(n, T, u)
    o.step(steps)
    with RLB(shape, order=order, eta_over_s=0.1) as g:
        g.init(n, T, u)
        g.step(steps)
        if o.nonconv:  # the model itself has cells without a frame: both stream them
            with pytest.raises(RLBError) as e:
                g.sync()
            assert e.value.status == RLB_ENONCONV and str(e.value).startswith("RLB_ENONCONV: %d cell" % o.nonconv)
            return g.populations(), None, o
        return g.populations(), g.moments(), o


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("scale", [1e-12, 1e-3, 1.0, 1e7, 1e20])
@pytest.mark.parametrize("vmax", [0.05, 0.8])
def test_double_steps_at_every_scale(order, scale, vmax):
    """The grid of the integer sums follows the populations' size; below and above the float range
    of the frame's first solve (1e-15, 1e15) the double iteration takes over.  1e-12 of each
    population's scale, as in the other double tests."""
    lat = oracle.read_lattice(order)
    n, T, u = gen.smooth_random_fields((6, 7, 18), seed=91, vmax=vmax, sigma_lnT=0.15, kmax=1, density="uniform")
    n = n * scale
    f, m, o = pair(lat, order, n, T, u, 2)
    ref = np.maximum(np.abs(o.f), lat.w[:, None, None, None] * n.max() / 2)
    assert np.max(np.abs(f - o.f) / ref) < 1e-12
    if m is None:
        return
    rn, reps, rU, _ = o.moments()
    assert np.max(np.abs(m["n"] - rn) / rn) < 1e-12
    assert np.max(np.abs(m["U"] - rU)) < 1e-12 * rU[0].max()


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("v", [0.9, 0.96, 0.975, 0.99])
def test_boosted_uniform_state_takes_the_double_iteration(order, v):
    """Below and above the Lorentz factor (4, v = 0.968) at which the frame is solved by the double
    iteration alone.  A boosted uniform equilibrium is stationary; the Landau solve and the
    equilibrium's cubic lose up to gamma^2 each to cancellation: 1e-12 gamma^4."""
    lat = oracle.read_lattice(order)
    shape = (4, 5, 6)
    n, T, u = np.ones(shape), np.ones(shape), np.zeros((3,) + shape)
    u[0], u[1], u[2] = 0.6 * v, 0.64 * v, 0.48 * v
    _, m, o = pair(lat, order, n, T, u, 1)
    assert m is not None
    g2 = 1 / (1 - v * v)
    assert np.max(np.abs(m["n"] - 1)) < 1e-12 * g2 ** 2
