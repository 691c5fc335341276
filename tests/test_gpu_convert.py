"""Population conversion in 16-byte units and its scalar remainder: sizes and pointers off the units."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB  # noqa: E402


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 3), (3, 5, 7), (2, 3, 4), (5, 9, 33)])
@pytest.mark.parametrize("offset", [0, 1])
def test_populations_round_trip(storage, shape, offset):
    """Device and host paths hand back what was set, rounded once to the storage type; `offset` moves
    the caller's array one double off a 16-byte boundary."""
    rng = np.random.default_rng(3)
    with RLB(shape, order=2, storage=storage) as g:
        n = g.q * g.cells
        f = rng.standard_normal((g.q,) + shape)
        want = f.astype(np.float32).astype(np.float64) if storage == "f32" else f
        buf = torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")
        view = buf[offset:offset + n].view(f.shape)
        view.copy_(torch.from_numpy(f))
        g.set_populations(view)
        view.zero_()
        g.populations(out=view)
        assert np.array_equal(view.cpu().numpy(), want)
        assert float(buf[n + 1]) == 7.0 and float(buf[0 if offset else n]) == 7.0
        assert np.array_equal(g.populations(), want)
        g.set_populations(f)
        assert np.array_equal(g.populations(), want)
