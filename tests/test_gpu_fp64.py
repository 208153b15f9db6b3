"""The FP64 kernels of the fine levels (half sweep, restriction, outer residual,
body force) against the oracle on ragged rows, walls of every kind and the
smoother's options; near_list_cells = 1 keeps every level out of the cluster
launch of the coarse ones."""
import numpy as np
import pytest

import oracle
import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W
from _pair import Pair, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,periodic,levels,nu1,nu2,omega", [
    ((42, 24, 36), (0, 1, 1), 2, 2, 2, 1.0),    # 21 cells a row on the coarser level
    ((36, 20, 26), (1, 1, 0), 2, 2, 2, 1.4),    # 18: no whole warp
    ((24, 20, 28), (0, 0, 0), 2, 0, 1, 1.0),    # from zero without a pre-smoothing
    ((136, 20, 24), (1, 0, 1), 3, 1, 2, 1.0),   # rows of several chunks
])
def test_fp64_cycle_and_body_force(dims, periodic, levels, nu1, nu2, omega):
    """The same iteration up to the rounding of sums of seven terms, a
    reciprocal for a division and, after a Gauss-Seidel sweep, black residuals
    of rounding size left out: 1e-14 an operation, 1e-12 after three cycles."""
    wl = W.mixed_box(dims=dims, periodic=periodic, levels=levels, n_spheres=3, radius=3.2)
    wl.omega, wl.nu1, wl.nu2, wl.coarse_sweeps = omega, nu1, nu2, 12
    p = Pair(wl, lib_overrides=dict(near_list_cells=1))
    p.o.map_particles()
    p.g.map_particles()
    fluid = p.o.owner() < 0
    for _ in range(3):
        io = p.o.solve(forced_cycles=1)
        ig = p.g.solve(forced_cycles=1)
        assert abs(ig["r0"] - io["r0"]) <= 1e-12 * io["r0"]
    assert rel_l2(p.g.field(es.FIELD_PSI)[fluid], p.o.field(oracle.FIELD_PSI)[fluid]) < 1e-12
    p.o.body_force()
    fb = p.g.field(es.FIELD_FB)
    assert rel_l2(fb[:, fluid], p.o.field(oracle.FIELD_FB)[:, fluid]) < 1e-12
    assert np.all(fb[:, ~fluid] == 0.0)


@pytest.mark.parametrize("dims,levels,lists", [((24, 20, 28), 1, 1), ((40, 36, 44), 1, 0), ((24, 20, 28), 1, 0),
                                               ((24, 20, 28), 2, 0)])
def test_mappings_in_a_row(dims, levels, lists):
    """Mappings that follow each other at once, with and without a move between:
    the oracle's owners every time (whole numbers).  One level
    with and without the cluster launch (40 x 36 x 44 is too large for it)."""
    wl = W.mixed_box(dims=dims, periodic=(1, 1, 0), levels=levels, n_spheres=3, radius=3.2)
    p = Pair(wl, lib_overrides=dict(near_list_cells=lists))
    rng = np.random.Generator(np.random.PCG64(5))
    for k in range(12):
        for _ in range(1 + k % 3):
            p.g.map_particles()
        p.o.map_particles()
        np.testing.assert_array_equal(p.g.field(es.FIELD_OWNER), p.o.owner())
        x = wl.x + rng.uniform(-0.3, 0.3, wl.x.shape)
        p.g.set_particles(x, wl.v, wl.w)
        p.o.set_particles(x, wl.v, wl.w)
        p.g.map_particles()
        p.g.map_particles()
        p.o.map_particles()
        np.testing.assert_array_equal(p.g.field(es.FIELD_OWNER), p.o.owner())
