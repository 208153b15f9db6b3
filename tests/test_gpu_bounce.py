"""Moving bounce-back of the FP64 stream-collide, one surface velocity a cell,
against the oracle's lever arm for each direction."""
import numpy as np
import pytest

import oracle
import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W
from _pair import Pair, rel_l2, to_oracle_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,periodic,x,radius", [
    ((20, 24, 20), (1, 1, 0), [[6.3, 7.1, 9.8], [13.6, 7.4, 10.2]], 3.2),   # cells next to two spheres
    ((16, 16, 16), (1, 1, 1), [[0.4, 8.2, 15.7]], 6.9),                     # two cells from the sphere's own image
    ((18, 16, 20), (1, 0, 1), [[17.6, 4.4, 0.3], [8.7, 11.2, 10.1]], 3.7),  # across the faces, near walls
])
def test_moving_bounce_back(dims, periodic, x, radius):
    """The same sums in another order, operands of order 0.1 and 19 terms a
    population: below 1e-15 each, 1e-13 of the field after two steps."""
    wl = W.mixed_box(dims=dims, periodic=periodic, n_spheres=len(x), radius=2.0, levels=1)
    wl.x, wl.R = np.array(x), np.full(len(x), radius)
    p = Pair(wl)
    for _ in range(2):
        for s in (p.o, p.g):
            s.map_particles()
            s.solve(forced_cycles=1)
        p.o.body_force()
        p.o.lbm_step()
        p.g.lbm_step()
    fluid = p.o.owner() < 0
    f, fo = to_oracle_order(p.g.field(es.FIELD_PDF)), p.o.field(oracle.FIELD_PDF)
    assert rel_l2(f[:, fluid] - fo[:, fluid] + 1.0, np.ones_like(fo[:, fluid])) < 1e-13
    assert np.max(np.abs(f[:, fluid] - fo[:, fluid])) < 1e-13
