"""Force and torque by momentum exchange: a block a sphere, with the box's rows
as bit words (R <= 13) or from the fields, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _workload(dims, periodic, radius, n, seed=7):
    wl = W.mixed_box(dims=dims, periodic=periodic, n_spheres=n, radius=radius, levels=2, seed=seed)
    wl.res_rf = 1e-8
    return wl


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32])
@pytest.mark.parametrize("dims,periodic,radius,n", [
    ((24, 20, 24), (1, 1, 1), 0.9, 3),      # a handful of cells
    ((16, 16, 20), (1, 1, 1), 6.2, 1),      # the box spans the whole axes
    ((32, 28, 32), (1, 0, 0), 3.3, 2),      # against walls
    ((32, 32, 32), (1, 1, 1), 12.9, 1),     # the longest rows of bit words
    ((36, 36, 36), (1, 1, 0), 14.2, 1),     # beyond them
    ((96, 96, 96), (1, 1, 1), 2.6, 330),    # many spheres: small blocks
])
def test_forces_match_oracle(precision, dims, periodic, radius, n):
    """FP64: the oracle's sums in another order, about 1e-15 of a cancelling
    sum: 1e-11.  MIXED32: the parity bar of the reduced forms, 1e-4."""
    wl = _workload(dims, periodic, radius, n)
    g, o = es.Simulation(wl, precision), oracle.Oracle(wl, omp=True)
    for _ in range(2):
        o.map_particles()
        info = o.solve()
        o.body_force()
        o.lbm_step()
        Fo, To = o.forces()
        o.advance()
        g.map_particles()
        g.solve(forced_cycles=info["cycles"] if precision == es.ES_FP64 else -1)
        g.lbm_step()
        F, T = g.forces()
        g.advance()
    tol = 1e-11 if precision == es.ES_FP64 else 1e-4
    assert np.linalg.norm(F - Fo) <= tol * np.linalg.norm(Fo)
    assert np.linalg.norm(T - To) <= tol * max(np.linalg.norm(To), radius * np.linalg.norm(Fo) * 0.1)
    g.close()


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32])
@pytest.mark.parametrize("dims,periodic,radius,shift", [
    ((16, 16, 20), (1, 1, 1), 6.9, (0.4, -0.3, 0.2)),  # a box as long as two axes allow
    ((16, 24, 16), (1, 0, 1), 6.8, (-0.4, 0.1, 0.45)),
    ((32, 32, 32), (1, 1, 1), 14.4, (0.3, 0.3, -0.4)),  # rows beyond the bit words
])
def test_forces_of_a_sphere_moved_since_its_mapping(precision, dims, periodic, radius, shift):
    """Momentum exchange with the links of the last mapping and the present centre:
    each surface cell is taken at its own nearest image, also where its fluid
    cell lies past half the axis.  Tolerances as above."""
    wl = _workload(dims, periodic, radius, 1)
    wl.x = np.array([[d / 2.0 + 0.2 for d in dims]])
    wl.v, wl.w = np.array([[0.02, -0.01, 0.015]]), np.array([[0.01, 0.02, -0.015]])
    g, o = es.Simulation(wl, precision), oracle.Oracle(wl)
    for s in (o, g):
        s.map_particles()
        s.solve(forced_cycles=1)
    o.body_force()
    for s in (o, g):
        s.lbm_step()
        s.set_particles(wl.x + np.array([shift]), wl.v, wl.w)
    Fo, To = o.forces()
    F, T = g.forces()
    tol = 1e-11 if precision == es.ES_FP64 else 1e-4
    assert np.linalg.norm(F - Fo) <= tol * np.linalg.norm(Fo)
    assert np.linalg.norm(T - To) <= tol * max(np.linalg.norm(To), radius * np.linalg.norm(Fo) * 0.1)
    g.close()


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32])
@pytest.mark.parametrize("n_small,big", [(0, 16.0), (340, 16.0), (340, 13.1)])
def test_forces_from_the_fields(precision, n_small, big):
    """A sphere whose rows are beyond the bit words, alone (1,024 threads a block)
    and among many small ones (256); tolerances as above."""
    dims = (88, 80, 72)
    wl = _workload(dims, (1, 1, 1), 2.6, 1)
    c = np.array([44.3, 40.1, 35.8])
    grid = np.array([(x, y, z) for x in range(4, 88, 8) for y in range(4, 80, 8) for z in range(4, 72, 8)], dtype=float)
    grid = grid[np.linalg.norm(grid - c, axis=1) > big + 5.0][:n_small]
    assert len(grid) == n_small
    n = 1 + n_small
    rng = np.random.Generator(np.random.PCG64(2))
    W._set_particles(wl, np.vstack([c[None], grid + 0.3]), np.array([big] + [2.6] * n_small),
                     np.array([i % 2 for i in range(n)]), np.ones(n), np.full(n, 1.3))
    wl.v, wl.w = rng.uniform(-0.02, 0.02, (n, 3)), rng.uniform(-0.01, 0.01, (n, 3))
    g, o = es.Simulation(wl, precision), oracle.Oracle(wl, omp=True)
    for s in (o, g):
        s.map_particles()
        s.solve(forced_cycles=1)
    o.body_force()
    for s in (o, g):
        s.lbm_step()
    Fo, To = o.forces()
    F, T = g.forces()
    tol = 1e-11 if precision == es.ES_FP64 else 1e-4
    for k in (slice(0, 1), slice(1, n)):  # the large one, and the others
        assert np.linalg.norm(F[k] - Fo[k]) <= tol * np.linalg.norm(Fo[k])
        assert np.linalg.norm(T[k] - To[k]) <= tol * max(np.linalg.norm(To[k]), 2.6 * np.linalg.norm(Fo[k]) * 0.1)
    g.close()
