"""Second-order double storage on the pipelined shapes with three and four consumer groups: they exist,
alone and in a batch, and step as the register kernel does, bit for bit (the double kernels add the same
integer sums)."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, Batch  # noqa: E402

# row segments take any x; row tiles a periodic x of at most 128 (16) or 96 cells (19)
CASES = [(15, (11, 13, 72), (0, 0, 0)), (15, (11, 13, 72), (1, 2, 0)), (15, (5, 7, 256), (2, 0, 1)),
         (16, (11, 13, 72), (0, 1, 2)), (16, (40, 32, 128), (0, 0, 0)), (19, (11, 13, 40), (0, 2, 0)),
         (19, (30, 31, 96), (0, 0, 0))]


@pytest.mark.parametrize("variant,shape,bc", CASES)
def test_shape_equals_register_kernel(variant, shape, bc):
    f = gen.smooth_random_fields(shape, seed=140, vmax=0.4, sigma_lnT=0.15, kmax=1)
    got = []
    for v in (variant, 0):
        with RLB(shape, order=2, bc=bc, step_variant=v) as g:
            assert g.variant == v
            g.init(*f)
            g.step(4)
            g.sync()
            got.append(g.populations())
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("variant", [15, 16, 19])
def test_batch_takes_the_shape(variant):
    with Batch(2, "f64") as b:
        b.set_variant(variant)
