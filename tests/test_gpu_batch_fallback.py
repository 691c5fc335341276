"""Members of a batch that its pipelined variant cannot take run as a context of their size runs alone: a
tube on the team kernel, a large box of odd rows on the register kernels, beside a pipelined box."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, Batch  # noqa: E402

MEMBERS = [((700, 1, 1), (0, 0, 1), 9), ((50, 51, 53), (0, 2, 0), 7), ((8, 16, 128), (0, 0, 0), 8),
           ((49, 49, 51), (0, 0, 0), 5)]


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage,variant,large", [("f32", 16, 3), ("f16dev", 12, 2), ("f64", 11, 0)])
@pytest.mark.parametrize("graph", [True, False])
def test_members_take_the_kernel_of_their_size(order, storage, variant, large, graph):
    ctxs = []
    for k, (shape, bc, steps) in enumerate(MEMBERS):
        f = gen.smooth_random_fields(shape, seed=150 + k, vmax=0.3, sigma_lnT=0.1, kmax=1)
        c = RLB(shape, order=order, bc=bc, storage=storage)
        c.init(*f)
        ctxs.append((c, f))
    with Batch(order, storage) as b:
        b.set_variant(variant)
        slots = [b.add(c, MEMBERS[k][2]) for k, (c, _) in enumerate(ctxs)]
        used = [b.member_variant(s) for s in slots]
        # the second member has 135,150 cells, the last 122,451: more than the team kernel's 116,736
        assert used == [20 if storage != "f64" else 0, large, variant, large]
        while b.run(4, graph=graph):
            pass
    for k, ((c, f), v) in enumerate(zip(ctxs, used)):
        shape, bc, steps = MEMBERS[k]
        with RLB(shape, order=order, bc=bc, storage=storage, step_variant=v) as s:
            assert s.variant == v
            s.init(*f)
            s.step(steps)
            assert np.array_equal(s.populations(), c.populations()), k
        c.close()
