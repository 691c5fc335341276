"""The extended-precision update of a float readout's Landau frame, apart from the error of the moments: the
same float populations read with the float solve and its update, and with every frame solved in double."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB  # noqa: E402


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage", ["f32", "f16dev"])
def test_updated_float_frame_equals_double_frame(order, storage):
    """Populations off equilibrium by 1e-3, so that T's anisotropy, the factor by which one update takes the
    frame nearer, is at most 4e-3.  The float solve is right to 1e-6 U0 (it stops at 3e-7; rounding of T.U);
    one update leaves 4e-9.  Without it, or with its residual in float, U would be off by a float rounding,
    6e-8.  n = U.N and eps = U.T.U follow U."""
    lat = oracle.read_lattice(order)
    rng = np.random.default_rng(31)
    shape = (3, 7, 9)
    f = np.empty((lat.q,) + shape)
    for c in np.ndindex(*shape):
        d = rng.standard_normal(3)
        v = 0.5 * rng.random()
        U = np.append(1.0, v * d / np.linalg.norm(d)) / np.sqrt(1 - v * v)
        f[(slice(None),) + c] = oracle.equilibrium_cell(lat, 0.8 + 0.4 * rng.random(), 1.0, U)
    f *= 1 + 1e-3 * rng.uniform(-1, 1, f.shape)
    got = []
    for fp64 in (False, True):
        with RLB(shape, order=order, storage=storage, landau_fp64=fp64) as g:
            g.set_populations(f)
            got.append(g.moments())
    a, b = got
    assert np.array_equal(a["totals"], b["totals"])  # the same moments
    assert np.max(np.abs(a["U"] - b["U"]) / b["U"][0]) < 4e-9
    assert np.max(np.abs(a["n"] / b["n"] - 1)) < 4e-9
    assert np.max(np.abs(a["eps"] / b["eps"] - 1)) < 4e-9
    uu = a["U"][0] ** 2 - (a["U"][1:] ** 2).sum(axis=0)
    assert np.max(np.abs(uu - 1)) < 1e-12
