"""Float initial states far from T = n = 1: populations that a float can hold come out finite and within float
rounding of the double ones, also where powers of T or n / T on the way to them leave the float range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB  # noqa: E402


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("T,n", [(1.0, 1.0), (1e8, 1.0), (1e10, 1.0), (1e13, 1.0), (1e15, 1e-5), (1e-8, 1.0),
                                 (1e-10, 1.0), (1e-39, 1e-10), (1.0, 1e-28), (1.0, 1e28)])
@pytest.mark.parametrize("v", [0.0, 0.5])
def test_float_initial_state_at_every_scale(order, T, n, v):
    """At rest: 32 roundings of 2^-24 of each population, three multiply-adds whose terms at the levels that are
    evaluated in float are up to ten times the value, on coefficients that are rounded once.  In motion a
    population may be a small difference of its terms, so only that it is finite."""
    shape = (2, 3, 43)
    u = np.zeros((3,) + shape)
    u[0], u[1], u[2] = 0.6 * v, -0.64 * v, 0.48 * v
    f = {}
    for storage in ("f32", "f64"):
        with RLB(shape, order=order, storage=storage) as g:
            g.init(np.full(shape, n), np.full(shape, T), u)
            f[storage] = g.populations()
    assert np.abs(f["f64"]).max() < 3e38 and np.all(np.isfinite(f["f32"]))
    if v > 0:
        return
    scale = np.abs(f["f64"]).max(axis=(1, 2, 3), keepdims=True) + 2.0 ** -126
    assert np.max(np.abs(f["f32"] - f["f64"]) / scale) < 32 * 2.0 ** -24
