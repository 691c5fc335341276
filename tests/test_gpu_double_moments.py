"""The moments of double populations (integer sums on a grid per energy level) at Lorentz factors from 1
to 4, where a few populations outgrow the others of their level: against sums in extended precision."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1301_3423_gb300.rlb import totals_noalloc  # noqa: E402


def sums(lat, f, kind):
    """N^0, T^00, T^0a of f (states, q), the terms added one after another in arithmetic `kind`."""
    f = f.astype(kind)
    p, v = lat.p0.astype(kind), lat.v.astype(kind) / np.sqrt(kind(lat.R2))
    out = np.zeros((5, len(f)), dtype=kind)
    for i in range(lat.q):
        out[0] += p[i] * f[:, i]
        out[1] += p[i] * p[i] * f[:, i]
        for a in range(3):
            out[2 + a] += p[i] * p[i] * v[i, a] * f[:, i]
    return out


@pytest.mark.parametrize("order", [3, 2])
@pytest.mark.parametrize("gamma", [1.0, 1.5, 2.0, 3.0, 4.0])
def test_moments_are_no_less_accurate_than_double_sums(order, gamma):
    """96 near-equilibrium states in random directions, one after another as a lattice of one cell, whose
    totals are its moments.  R.m.s. error relative to T^00 (N^0 for N^0) against that of adding the 128
    terms in double; a quarter more is what the scatter of 480 samples can make of equal errors."""
    lat = oracle.read_lattice(order)
    rng = np.random.default_rng(17)
    states = []
    for _ in range(96):
        d = rng.standard_normal(3)
        U = np.append(gamma, np.sqrt(gamma * gamma - 1) * d / np.linalg.norm(d))
        f = oracle.equilibrium_cell(lat, 1.0 + rng.random(), 1.0, U)
        states.append(f * (1 + 1e-3 * rng.standard_normal(lat.q)))
    states = np.array(states)
    got = [totals_noalloc(torch.from_numpy(f).cuda(), order, "f64", (1, 1, 1)) for f in states]
    ref = sums(lat, states, np.longdouble)
    scale = np.stack([ref[0], ref[1], ref[1], ref[1], ref[1]])
    rms = [float(np.sqrt(np.mean(np.square((x - ref) / scale)))) for x in (np.array(got).T, sums(lat, states, np.float64))]
    print("order %d gamma %g: %.2e, double sums %.2e" % (order, gamma, *rms))
    assert rms[0] <= 1.25 * rms[1]
