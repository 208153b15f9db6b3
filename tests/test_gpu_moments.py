"""Density and velocity read back from the reduced forms: float-float sums of
the stored deviations against FP64 sums of the populations read back."""
import numpy as np
import pytest

import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32, es.ES_MIXED16])
@pytest.mark.parametrize("dims,periodic", [((42, 24, 32), (0, 1, 1)), ((40, 24, 32), (1, 1, 0)), ((24, 36, 20), (1, 1, 1))])
def test_moments_match_populations(precision, dims, periodic):
    """FP64 sums of 19 populations below 1/3 round by at most 19 x 2^-53; the
    float-float sums drop below 2^-46 of the deviations (< 0.1): 4e-15."""
    wl = W.mixed_box(dims=dims, periodic=periodic, levels=2)
    wl.accel = (1e-4, -2e-4, 3e-4)
    sim = es.Simulation(wl, precision)
    for _ in range(3):
        sim.step()
    u, rho = sim.field(es.FIELD_U), sim.field(es.FIELD_RHO)  # (before f_b itself is read)
    f, fb = sim.field(es.FIELD_PDF), sim.field(es.FIELD_FB)
    c, _ = es.lattice()
    want = np.stack([sum(c[q][a] * f[q] for q in range(19) if c[q][a]) for a in range(3)])
    want -= 0.5 * (fb + np.array(wl.accel).reshape(3, 1, 1, 1))
    assert np.abs(f - f.mean(axis=(1, 2, 3), keepdims=True)).max() < 0.1
    np.testing.assert_allclose(u, want, rtol=0, atol=4e-15)
    np.testing.assert_allclose(rho, f.sum(0), rtol=0, atol=4e-15)
    sim.close()


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32, es.ES_MIXED16])
def test_moments_of_infinite_populations(precision):
    """A diverged state reads back as the FP64 sums of its populations would:
    infinities keep their sign, opposite ones give NaN."""
    wl = W.mixed_box(dims=(24, 20, 16), periodic=(1, 1, 1), levels=2)
    sim = es.Simulation(wl, precision)
    sim.step()
    f = sim.field(es.FIELD_PDF)
    c, _ = es.lattice()
    east, west = (next(q for q in range(19) if tuple(c[q]) == v) for v in ((1, 0, 0), (-1, 0, 0)))
    cells = [(1, 2, 3), (4, 5, 6), (7, 8, 9)]
    f[(east,) + cells[0]] = np.inf
    f[(west,) + cells[1]] = np.inf
    f[(east,) + cells[2]], f[(west,) + cells[2]] = np.inf, -np.inf
    sim.set_field(es.FIELD_PDF, f)
    rho, u = sim.field(es.FIELD_RHO), sim.field(es.FIELD_U)
    assert rho[cells[0]] == np.inf and rho[cells[1]] == np.inf and np.isnan(rho[cells[2]])
    assert u[0][cells[0]] == np.inf and u[0][cells[1]] == -np.inf and u[0][cells[2]] == np.inf
    rest = np.ones(rho.shape, dtype=bool)
    for k in cells:
        rest[k] = False
    assert np.isfinite(rho[rest]).all() and np.isfinite(u[:, rest]).all()
    sim.close()
