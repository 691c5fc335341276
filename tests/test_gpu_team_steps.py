"""Several steps of a small lattice in one cooperative launch: every order, boundary kind and storage, more
tiles than the device holds blocks, the barrier's bounded wait, and a grid that does not fit."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, RLBError  # noqa: E402
from paper_1301_3423_gb300 import rlb as rlbmod  # noqa: E402

TEAM = rlbmod.VARIANT_NAMES.index("team 4x32")
SMALL = ((10, 31, 33), (1, 0, 2))
# 64,050 to 108,000 cells: two to four tiles for each of the 912 blocks that hold float tiles
LARGE = [((50, 21, 61), (0, 2, 0)), ((50, 48, 45), (1, 0, 0))]


def fields(shape, seed):
    return gen.smooth_random_fields(shape, seed=seed, vmax=0.3, sigma_lnT=0.1, kmax=1)


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage,shape,bc", [(s, *SMALL) for s in ("f64", "f32", "f16dev")]
                         + [(s, *c) for s in ("f32", "f16dev") for c in LARGE]
                         + [("f64", (97, 1, 1), (0, 0, 2)), ("f32", (31, 1, 1), (0, 0, 2))])
def test_several_steps_equal_single_steps(order, storage, shape, bc):
    f = fields(shape, 160)
    got, launches = [], []
    for v in (-1, TEAM):
        with RLB(shape, order=order, bc=bc, storage=storage, step_variant=v) as g:
            assert g.variant == TEAM
            g.init(*f)
            n0 = g.kernel_launches
            g.step(67)
            g.sync()
            launches.append(g.kernel_launches - n0)
            got.append((g.populations(), g.moments()["U"]))
    assert launches == [2, 67]
    assert all(np.array_equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_expired_barrier_is_reported_and_the_context_stays_usable(storage):
    """Testing flag: the barrier waits for one block more than the grid has.  Every block's wait (2 s) runs
    out, the kernel returns, and the context works again once a state is restored."""
    shape = (97, 3, 1)
    with RLB(shape, bc=(0, 0, 1), storage=storage, debug_flags=4) as g:
        assert g.variant == TEAM
        g.init(*fields(shape, 161))
        f0 = g.populations()
        g.step(3)
        with pytest.raises(RLBError) as e:
            g.sync()
        assert e.value.status == rlbmod.RLB_ETIMEOUT
        g.sync()  # reported once
        g.set_populations(f0)
        g.step(1)  # one step needs no barrier
        g.sync()
        with RLB(shape, bc=(0, 0, 1), storage=storage) as h:
            h.set_populations(f0)
            h.step(1)
            assert np.array_equal(g.populations(), h.populations())


def test_a_grid_that_does_not_fit_takes_single_steps():
    """Testing flag: the launch asks for twice the blocks that the device holds and is refused; the same
    steps are taken one launch each, and every later one too."""
    shape, bc = LARGE[0]
    f = fields(shape, 162)
    got = []
    for flags in (2, 0):
        with RLB(shape, bc=bc, storage="f32", debug_flags=flags) as g:
            assert g.variant == TEAM
            g.init(*f)
            n0 = g.kernel_launches
            g.step(5)
            g.step(4)
            g.sync()
            assert g.kernel_launches - n0 == (9 if flags else 2) and g.steps_done == 9
            got.append(g.populations())
    assert np.array_equal(*got)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_several_steps_in_a_captured_graph(storage):
    """A captured launch of several steps replays as the same steps taken directly."""
    shape, bc = SMALL
    f = fields(shape, 163)
    s = torch.cuda.Stream()
    with RLB(shape, bc=bc, storage=storage, stream=s) as g, RLB(shape, bc=bc, storage=storage) as h:
        assert g.variant == TEAM
        g.init(*f)
        h.init(*f)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            g.step(6)  # an even number: the state ends in the buffer it began in
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        h.step(18)
        assert np.array_equal(g.populations(), h.populations())
