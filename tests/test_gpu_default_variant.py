"""The step variant the library chooses by itself, on both sides of each line of its rule."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB  # noqa: E402

TEAM = 20
# (shape (nz, ny, nx), bc (x, y, z), order, variant float, half)
CASES = [
    # rows that fill a slower tile and leave some of a faster one
    ((40, 41, 40), (0, 0, 0), 3, 16, 23), ((40, 41, 40), (0, 0, 0), 2, 16, 23), ((80, 80, 72), (0, 0, 0), 3, 21, 23),
    ((80, 80, 24), (0, 0, 0), 3, 22, 22), ((40, 40, 160), (0, 0, 0), 3, 21, 21), ((40, 40, 176), (0, 0, 0), 3, 22, 22),
    # an x that is not periodic: no segments, however many
    ((20, 20, 640), (1, 0, 0), 3, 3, 2), ((20, 20, 640), (2, 0, 0), 2, 3, 2), ((16, 16, 1024), (1, 0, 0), 3, 3, 2),
    ((20, 20, 640), (0, 0, 0), 3, 15, 15),
    # walls on y or z near one row in eight, in 19 and in 21
    ((40, 96, 96), (0, 2, 0), 3, 3, 2), ((96, 40, 96), (0, 0, 2), 3, 3, 2), ((6, 232, 128), (0, 2, 0), 3, 3, 2),
    ((6, 256, 128), (0, 2, 0), 3, 16, 23),
    ((24, 24, 24), (0, 2, 0), 3, TEAM, TEAM), ((20, 20, 256), (0, 2, 0), 3, TEAM, TEAM),
    # segments 5/6 used
    ((20, 24, 320), (0, 0, 0), 3, 15, 15), ((20, 24, 320), (0, 0, 0), 2, 15, 2),
    # the largest lattices of the team kernel: 116,736 cells
    ((46, 49, 51), (0, 0, 0), 3, TEAM, TEAM), ((46, 49, 48), (1, 0, 0), 3, TEAM, TEAM), ((47, 49, 51), (0, 0, 0), 3, 3, 2),
]


@pytest.mark.parametrize("shape,bc,order,f32,f16", CASES)
def test_default_variant(shape, bc, order, f32, f16):
    for storage, want in (("f32", f32), ("f16dev", f16)):
        with RLB(shape, order=order, bc=bc, storage=storage) as g:
            assert g.variant == want, storage
