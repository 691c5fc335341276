"""The wide row tiles (160, 192 and 256 cells), and row segments refilled in chunks: against the other
tilings of the same pulls, bit for bit."""
import numpy as np
import pytest

from paper_inputs import fields as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300 import RLB, Batch  # noqa: E402

# (shape (nz, ny, nx), bc): rows that fill a wide tile alone, several to a tile, a short last tile, wraps
# of y and z inside a tile, open and walled y and z
CASES = [((7, 9, 160), (0, 0, 0)), ((5, 13, 192), (0, 0, 0)), ((4, 7, 256), (0, 1, 0)), ((9, 11, 40), (0, 0, 0)),
         ((13, 7, 64), (0, 2, 1)), ((6, 10, 96), (0, 0, 2)), ((5, 30, 8), (0, 0, 0)), ((20, 16, 128), (0, 0, 0)),
         ((3, 5, 176), (0, 2, 2))]


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("storage", ["f32", "f16dev"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_wide_row_tiles_equal_row_segments(order, storage, case):
    shape, bc = CASES[case]
    n, T, u = gen.smooth_random_fields(shape, seed=110 + case, vmax=0.4, sigma_lnT=0.15, kmax=1)
    got = {}
    for v in (15, 21, 22, 23):
        with RLB(shape, order=order, bc=bc, storage=storage, eta_over_s=0.1, step_variant=v) as g:
            if g.variant != v:
                assert v != 15
                continue
            g.init(n, T, u)
            g.step(5)
            got[v] = g.populations()
    assert len(got) >= 2 or shape[2] > 192
    for v in got:
        assert np.array_equal(got[v], got[15]), v


@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 0), (2, 2, 1)])
def test_chunked_segments_with_some_cells_without_a_frame(bc):
    """Warps some of whose cells have no Landau frame keep their stage whole (no early release).  NaN in
    a few cells leaves every cell that pulls from them without a frame: the same cells are counted and
    streamed as by the kernel that refills whole stages, the others agree to the order of the sums."""
    from paper_1301_3423_gb300 import RLBError
    shape = (40, 24, 256)
    n, T, u = gen.smooth_random_fields(shape, seed=121, vmax=0.3, sigma_lnT=0.1, kmax=1)
    got, counts = [], []
    for v in (15, 4):
        with RLB(shape, bc=bc, storage="f32", step_variant=v) as g:
            g.init(n, T, u)
            f = torch.empty((g.q,) + shape, dtype=torch.float64, device="cuda")
            g.populations(out=f)
            f[:, 5:9, 3, 60:90] = float("nan")
            g.set_populations(f)
            g.step(1)
            with pytest.raises(RLBError) as e:
                g.sync()
            counts.append(str(e.value))
            got.append(g.populations())
    assert counts[0] == counts[1]
    a, b = got
    assert np.array_equal(np.isnan(a), np.isnan(b))
    scale = np.nanmax(np.abs(b), axis=(1, 2, 3), keepdims=True)
    assert np.nanmax(np.abs(a - b) / scale) < 4e-6  # one and two warps per cell sum in another order


def test_chunked_segments_without_any_frame():
    """One population everywhere: every cell streams it unchanged, over several tiles per block.  Powers of
    two, so that a lone population's null current rounds alike in every cell."""
    from paper_1301_3423_gb300 import RLBError
    shape = (40, 24, 256)
    with RLB(shape, storage="f32", step_variant=15) as g:
        x = (2.0 ** np.random.default_rng(5).integers(-3, 4, shape)).astype(np.float32)
        f = torch.zeros((g.q,) + shape, dtype=torch.float64, device="cuda")
        f[0] = torch.from_numpy(x).cuda()
        g.set_populations(f)
        g.step(1)
        with pytest.raises(RLBError) as e:
            g.sync()
        assert "%d cell" % x.size in str(e.value)
        p = g.populations()
    from paper_1301_3423_gb300 import quadrature
    v = quadrature(3)["v"][0]
    assert np.array_equal(p[0], np.roll(x, (v[2], v[1], v[0]), axis=(0, 1, 2))) and not p[1:].any()


@pytest.mark.parametrize("variant", [21, 22, 23])
def test_batch_of_wide_row_tiles_equals_solo_runs(variant):
    shapes = [(8, 9, 40), (6, 5, 160), (7, 5, 192), (4, 5, 256), (9, 1, 1), (5, 7, 96)]
    with Batch(3, "f16dev") as b:
        b.set_variant(variant)
        ctxs, solo = [], []
        for k, shape in enumerate(shapes):
            f = gen.smooth_random_fields(shape, seed=130 + k, vmax=0.3, sigma_lnT=0.1, kmax=1)
            c = RLB(shape, storage="f16dev")
            c.init(*f)
            ctxs.append((c, b.add(c, 5 + k), f))
        used = [b.member_variant(s) for _, s, _ in ctxs]
        assert variant in used
        while b.run(4):
            pass
        for k, ((c, _, f), v) in enumerate(zip(ctxs, used)):
            with RLB(shapes[k], storage="f16dev", step_variant=v) as s:
                assert s.variant == v
                s.init(*f)
                s.step(5 + k)
                solo.append(np.array_equal(s.populations(), c.populations()))
            c.close()
        assert all(solo)
