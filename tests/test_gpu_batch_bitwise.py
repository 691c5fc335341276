"""A member of a batch on the register kernels takes the steps it would take alone bit for bit: every
variant, order and boundary kind, with odd rows, interior and boundary rows."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, Batch  # noqa: E402


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage,variant", [("f64", 0)] + [(s, v) for s in ("f32", "f16dev") for v in range(4)])
@pytest.mark.parametrize("bc", [(0, 0, 0), (0, 2, 0), (1, 0, 2)])
def test_register_member_equals_solo_run(order, storage, variant, bc):
    shape = (40, 41, 53)
    f = gen.smooth_random_fields(shape, seed=151, vmax=0.3, sigma_lnT=0.1, kmax=1)
    got = []
    for batched in (True, False):
        with RLB(shape, order=order, bc=bc, storage=storage, step_variant=variant) as c:
            assert c.variant == variant
            c.init(*f)
            if batched:
                with Batch(order, storage) as b:
                    b.set_variant(variant)
                    b.add(c, 2)
                    b.run(2)
            else:
                c.step(2)
            got.append(c.populations())
    assert np.array_equal(*got)
