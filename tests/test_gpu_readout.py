"""The fields readout of float contexts against a double context holding the same populations: the
pull offsets per axis (axes shorter than the stencil reach, odd sizes, every boundary) and the
float-float update of the Landau frame."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB  # noqa: E402

# (shape (nz, ny, nx), bc (x, y, z))
CASES = [((3, 5, 7), (0, 0, 0)), ((41, 1, 1), (0, 0, 1)), ((13, 2, 1), (0, 0, 2)), ((1, 1, 6), (0, 0, 0)),
         ((9, 12, 33), (1, 2, 0)), ((7, 13, 31), (2, 1, 2)), ((12, 20, 129), (0, 0, 0))]


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage", ["f32", "f16dev"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_float_readout_equals_double_readout_of_the_same_populations(order, storage, case):
    """After one step the readout pulls the populations from before it, which both contexts hold
    exactly; what differs is the float sums: at most 128 roundings of 2^-24 in each moment, whose
    terms are at most about the moment itself, and typically a tenth of that: 4e-6."""
    shape, bc = CASES[case]
    n, T, u = gen.smooth_random_fields(shape, seed=60 + case, vmax=0.4, sigma_lnT=0.15, kmax=1)
    with RLB(shape, order=order, bc=bc, storage=storage) as a, RLB(shape, order=order, bc=bc) as b:
        a.init(n, T, u)
        b.set_populations(a.populations())
        a.step(1)
        b.step(1)
        ma, mb = a.moments(), b.moments()
    for k in ("n", "eps"):
        assert np.max(np.abs(ma[k] - mb[k]) / mb[k]) < 4e-6
    assert np.max(np.abs(ma["U"] - mb["U"])) < 4e-6 * mb["U"][0].max()
    # U.U = 1 holds to the float-float arithmetic of the readout, not to float
    uu = ma["U"][0] ** 2 - (ma["U"][1:] ** 2).sum(axis=0)
    assert np.max(np.abs(uu - 1)) < 1e-12 * ma["U"][0].max() ** 2
    assert np.max(np.abs(ma["totals"] - mb["totals"])) < 4e-6 * np.abs(mb["totals"]).max()


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_device_outputs_written_in_place_equal_host_outputs(storage):
    """Device outputs, as views into one allocation at odd offsets with guard values around them, hold
    what the host path returns; so does one output alone."""
    import ctypes
    shape = (5, 9, 33)
    cells = 5 * 9 * 33
    n, T, u = gen.smooth_random_fields(shape, seed=75, vmax=0.4, sigma_lnT=0.15, kmax=1)
    with RLB(shape, storage=storage) as g:
        g.init(n, T, u)
        g.step(2)
        ref = g.moments()
        buf = torch.full((6 * cells + 10,), 7.0, dtype=torch.float64, device="cuda")
        out = dict(n=buf[1:1 + cells].view(shape), eps=buf[3 + cells:3 + 2 * cells].view(shape),
                   U=buf[5 + 2 * cells:5 + 6 * cells].view((4,) + shape))
        got = g.moments(out=out)
        for k in ("n", "eps", "U"):
            assert np.array_equal(got[k].cpu().numpy(), ref[k])
        guards = [0, 1 + cells, 2 + cells, 3 + 2 * cells, 4 + 2 * cells, 5 + 6 * cells]
        assert all(float(buf[k]) == 7.0 for k in guards)
        # one output alone (the others NULL)
        tot = (ctypes.c_double * 5)()
        buf.fill_(7.0)
        assert g._lib.rlb_moments(g._h, None, ctypes.c_void_p(out["eps"].data_ptr()), None, tot, 1) == 0
        assert np.array_equal(out["eps"].cpu().numpy(), ref["eps"]) and float(buf[1]) == 7.0
        assert np.array_equal(np.array(tot[:]), ref["totals"])
