"""The team kernel (four warps share 32 cells): against the register kernels over every boundary and
ragged tile, and several steps in one launch against the same steps one at a time."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, Batch  # noqa: E402
from paper_1301_3423_gb300 import rlb as rlbmod  # noqa: E402

TEAM = rlbmod.VARIANT_NAMES.index("team 4x32")
# (shape (nz, ny, nx), bc (x, y, z)): one cell, a tile short and over, axes below the stencil reach,
# walls and open ends, interior warps, several tiles per block of the cooperative launch
CASES = [((1, 1, 1), (0, 0, 0)), ((31, 1, 1), (0, 0, 1)), ((33, 1, 1), (0, 0, 2)), ((3, 5, 7), (0, 0, 0)),
         ((9, 12, 33), (1, 2, 0)), ((7, 13, 31), (2, 1, 2)), ((16, 15, 80), (0, 0, 0)), ((20, 70, 90), (0, 2, 1))]


def fields(shape, seed):
    return gen.smooth_random_fields(shape, seed=seed, vmax=0.3, sigma_lnT=0.1, kmax=1)


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage,reg,tol", [("f64", 0, 0.0), ("f32", 3, 4e-6), ("f16dev", 2, 4e-3)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_team_equals_register_kernel(order, storage, reg, tol, case):
    """Double: the same arithmetic per population and integer moments, bit for bit.  Float: the same
    but for the order of the moments' sums, a few 2^-24 a step over 5 steps, relative to the largest
    population of each kind; half stores that with roundings of 2^-11."""
    shape, bc = CASES[case]
    n, T, u = fields(shape, 70 + case)
    got = []
    for v in (TEAM, reg):
        with RLB(shape, order=order, bc=bc, storage=storage, step_variant=v) as g:
            assert g.variant == v
            g.init(n, T, u)
            g.step(5)
            got.append(g.populations())
    if tol == 0.0:
        assert np.array_equal(got[0], got[1])
    else:
        scale = np.abs(got[1]).max(axis=(1, 2, 3), keepdims=True)
        assert np.max(np.abs(got[0] - got[1]) / scale) < tol


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("steps", [2, 3, 65, 130])
def test_steps_in_one_launch_equal_single_steps(storage, steps):
    for shape, bc in (((97, 1, 1), (0, 0, 1)), ((30, 31, 33) if storage != "f64" else (10, 31, 33), (0, 0, 0))):
        n, T, u = fields(shape, 80)
        # the library's choice for such a lattice; asked for, it takes one launch per step
        with RLB(shape, bc=bc, storage=storage) as a, \
                RLB(shape, bc=bc, storage=storage, step_variant=TEAM) as b:
            assert a.variant == b.variant == TEAM
            a.init(n, T, u)
            b.init(n, T, u)
            la, lb = a.kernel_launches, b.kernel_launches
            a.step(steps)
            b.step(steps)
            assert a.kernel_launches - la == -(-steps // 64) and b.kernel_launches - lb == steps
            assert np.array_equal(a.populations(), b.populations())
            assert np.array_equal(a.moments()["n"], b.moments()["n"])


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_batch_of_team_members_equals_solo_runs(storage):
    shapes = [((400, 1, 1), (0, 0, 1)), ((3, 5, 7), (0, 0, 0)), ((9, 12, 33), (1, 2, 0))]
    ctxs = []
    for k, (shape, bc) in enumerate(shapes):
        c = RLB(shape, bc=bc, storage=storage)
        c.init(*fields(shape, 90 + k))
        ctxs.append(c)
    with Batch(3, storage) as b:
        b.set_variant(TEAM)
        for k, c in enumerate(ctxs):
            b.add(c, 7 + 4 * k)
        while b.run(6):
            pass
    for k, ((shape, bc), c) in enumerate(zip(shapes, ctxs)):
        with RLB(shape, bc=bc, storage=storage, step_variant=TEAM) as s:
            s.init(*fields(shape, 90 + k))
            s.step(7 + 4 * k)
            assert np.array_equal(s.populations(), c.populations())
        c.close()
