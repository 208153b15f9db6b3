"""The coarse levels of the V-cycle in one cluster launch against the same
levels launched one by one (near_list_cells = 1 keeps every level out of it)."""
import numpy as np
import pytest

import oracle
import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W
from _pair import rel_l2

pytestmark = pytest.mark.gpu

CASES = [  # dims, periodic, levels, nu1, nu2, omega
    ((32, 32, 32), (1, 1, 1), 3, 2, 2, 1.0),
    ((64, 64, 64), (1, 1, 1), 4, 2, 2, 1.0),
    ((64, 64, 64), (1, 1, 0), 5, 1, 2, 1.0),
    ((42, 24, 36), (0, 1, 1), 2, 2, 2, 1.0),   # 21 cells a row on the coarser level
    ((36, 44, 26), (1, 1, 0), 2, 2, 1, 1.0),
    ((48, 40, 56), (1, 1, 1), 3, 2, 0, 1.0),
    ((40, 24, 32), (0, 0, 0), 3, 1, 1, 1.3),
    ((128, 16, 24), (1, 1, 1), 3, 0, 2, 1.0),
    ((96, 96, 48), (1, 1, 0), 4, 2, 2, 1.0),   # only the coarser levels fit
    ((24, 20, 28), (1, 1, 1), 1, 2, 2, 1.7),   # one level: sweeps only
]


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32])
@pytest.mark.parametrize("dims,periodic,levels,nu1,nu2,omega", CASES)
def test_cluster_levels_match_separate_launches(precision, dims, periodic, levels, nu1, nu2, omega):
    """FP64: two V-cycles, the same iteration up to the rounding of a few sums
    (each below 1e-15 of the iterate, contracted by the cycle): 1e-12.
    MIXED32: both iterations end below 1e-10 of the first residual, so the
    potentials differ by at most 2e-10 cond(A) < 2e-10 (12 + kappa^2) / kappa^2 = 3e-8."""
    wl = W.mixed_box(dims=dims, periodic=periodic, levels=levels, n_spheres=3, radius=3.2)
    wl.omega, wl.nu1, wl.nu2, wl.coarse_sweeps, wl.max_cycles = omega, nu1, nu2, 12, 300
    out = []
    for lists in (0, 1):
        sim = es.Simulation(wl, precision, overrides=dict(near_list_cells=lists))
        sim.map_particles()
        sim.solve(forced_cycles=2 if precision == es.ES_FP64 else -1)
        out.append(sim.field(es.FIELD_PSI))
        sim.close()
    diff = np.linalg.norm(out[0] - out[1]) / np.linalg.norm(out[1])
    assert np.linalg.norm(out[1]) > 0
    assert diff < (1e-12 if precision == es.ES_FP64 else 3e-8), diff


@pytest.mark.parametrize("dims,levels", [((64, 64, 64), 4), ((128, 64, 64), 4), ((128, 128, 128), 4)])
def test_bulk_copied_right_hand_side(dims, levels):
    """Colour-split right-hand sides of whole spans come into the cluster by bulk
    copies over places that were zeroed: the same start gives the same bits
    every time."""
    wl = W.mixed_box(dims=dims, levels=levels, n_spheres=3, radius=3.2, periodic=(1, 1, 1))
    sim = es.Simulation(wl, es.ES_MIXED32)
    sim.map_particles()
    psi0 = np.zeros(dims[::-1])
    ref = None
    for _ in range(24):
        sim.set_field(es.FIELD_PSI, psi0)
        sim.solve(forced_cycles=2)
        psi = sim.field(es.FIELD_PSI)
        assert np.isfinite(psi).all() and np.linalg.norm(psi) > 0
        if ref is None:
            ref = psi
        np.testing.assert_array_equal(psi, ref)
    sim.close()


def _levels_in_cluster(sim):
    """The levels of the cluster launches of one V-cycle."""
    sim.profile_start()
    sim.solve(forced_cycles=1)
    return [r["level"] for r in sim.profile_stop() if r["name"] == "tail"]


@pytest.mark.parametrize("precision", [es.ES_FP64, es.ES_MIXED32])
@pytest.mark.parametrize("dims,axis", [((32, 32, 1), 0), ((64, 1, 1), 0), ((1, 32, 32), 1), ((1, 1, 40), 2),
                                       ((36, 1, 20), 2)])
def test_periodic_axis_of_one_cell(precision, dims, axis):
    """A cell is its own neighbour along a periodic axis of one cell.  FP64: the
    oracle's iteration up to the rounding of sums of seven terms, 1e-12 after
    two cycles, and its cycle count.  MIXED32: below 1e-10 of the first residual
    after one cycle more (FP32 reaches 1e-5 a cycle and more here), so the
    potentials differ by at most 2e-10 (12 + kappa^2) / kappa^2 = 3e-8."""
    bc, val = [0] * 6, [0.0] * 6
    bc[2 * axis] = bc[2 * axis + 1] = 1
    val[2 * axis], val[2 * axis + 1] = 0.7, -0.4
    wl = W.Workload(name="thin", dims=list(dims), periodic=tuple(0 if a == axis else 1 for a in range(3)), tau=0.8,
                    kappa=0.3, eps=1.0, E_ext=(0.0, 0.0, 0.0), levels=1, coarse_sweeps=400, res_rf=1e-10,
                    max_cycles=200, pot_bc=tuple(bc), pot_val=tuple(val))
    sim, o = es.Simulation(wl, precision), oracle.Oracle(wl)
    sim.map_particles()
    o.map_particles()
    if precision == es.ES_FP64:
        io, ig = o.solve(forced_cycles=2), sim.solve(forced_cycles=2)
        assert rel_l2(sim.field(es.FIELD_PSI), o.field(oracle.FIELD_PSI)) < 1e-12
        assert abs(ig["r0"] - io["r0"]) <= 1e-12 * io["r0"]
        assert sim.solve()["cycles"] == o.solve()["cycles"]
    else:
        io = o.solve()
        assert sim.solve(forced_cycles=io["cycles"] + 1)["r"] <= io["tol"]
        assert rel_l2(sim.field(es.FIELD_PSI), o.field(oracle.FIELD_PSI)) < 3e-8
    assert _levels_in_cluster(sim) == []
    sim.close()


@pytest.mark.parametrize("precision,dims,levels,lists,want", [
    (es.ES_FP64, (32, 32, 32), 3, 0, [1]),
    (es.ES_FP64, (24, 20, 28), 2, 0, [0]),
    (es.ES_MIXED32, (64, 64, 64), 4, 0, [0]),
    (es.ES_MIXED32, (96, 96, 48), 4, 0, [1]),
    (es.ES_MIXED32, (64, 64, 64), 4, 1, []),
])
def test_levels_of_the_cluster_launch(precision, dims, levels, lists, want):
    """The cluster launch runs, from the finest level that fits it on;
    near_list_cells = 1 keeps every level out of it."""
    wl = W.mixed_box(dims=dims, periodic=(1, 1, 1), levels=levels, n_spheres=3, radius=3.2)
    sim = es.Simulation(wl, precision, overrides=dict(near_list_cells=lists))
    sim.map_particles()
    assert _levels_in_cluster(sim) == want
    sim.close()


@pytest.mark.parametrize("dims,periodic,levels,nu1,nu2,omega", [c for c in CASES if c[5] == 1.0] + [
    ((40, 24, 32), (0, 0, 0), 2, 1, 1, 1.3),   # over-relaxed: colour-split level, coarsest level
    ((42, 24, 36), (0, 1, 1), 2, 2, 2, 0.8),   # and rows that are no whole spans
    ((24, 20, 28), (1, 1, 1), 1, 2, 2, 1.7),
])
def test_cluster_levels_give_the_same_bits(dims, periodic, levels, nu1, nu2, omega):
    """In FP32 the cluster launch does the operations of the separate launches in
    their order: the same potential to the last bit.  kappa = 0.37: diagonals
    that round when faces are added and taken away.  (Over-relaxed levels of
    whole spans that are not split round their near-boundary cells another way
    from the lists than inline, which the cluster follows.)"""
    wl = W.mixed_box(dims=dims, periodic=periodic, levels=levels, n_spheres=3, radius=3.2)
    wl.kappa, wl.omega, wl.nu1, wl.nu2, wl.coarse_sweeps = 0.37, omega, nu1, nu2, 12
    if not periodic[2]:
        wl.pot_bc, wl.pot_val = (0, 0, 0, 0, 1, 0), (0.0, 0.0, 0.0, 0.0, 0.3, 0.0)
    out = []
    for lists in (0, 1):
        sim = es.Simulation(wl, es.ES_MIXED32, overrides=dict(near_list_cells=lists))
        sim.map_particles()
        sim.solve(forced_cycles=2)
        out.append(sim.field(es.FIELD_PSI))
        sim.close()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("precision,dims,levels,want", [
    (es.ES_MIXED32, (64, 160, 16), 1, [0]),    # 10,240 cells of the coarsest level in each of 16 blocks
    (es.ES_MIXED32, (64, 168, 16), 1, []),
    (es.ES_MIXED32, (128, 128, 4), 1, []),     # four blocks
    (es.ES_MIXED32, (128, 128, 16), 2, [1]),   # 64 x 64 x 8
    (es.ES_MIXED32, (64, 64, 64), 2, [0]),     # above it 16,384 a block
    (es.ES_MIXED32, (64, 72, 56), 2, [1]),
    (es.ES_FP64, (32, 32, 16), 1, [0]),        # 1,024 cells
    (es.ES_FP64, (32, 34, 16), 1, []),
    (es.ES_FP64, (64, 64, 8), 1, []),
    (es.ES_FP64, (16, 32, 32), 2, [0]),
    (es.ES_FP64, (20, 28, 28), 2, [1]),        # (1,120)
    (es.ES_FP64, (96, 80, 12), 2, [1]),        # 48 x 40 x 6: one block would solve it
    (es.ES_FP64, (64, 64, 2), 1, [0]),
])
def test_flat_levels_are_launched(precision, dims, levels, want):
    """Which levels the cluster takes by the cells of a block's planes; the same
    V-cycle either way: the bits in FP32, 1e-12 in FP64 (as above)."""
    wl = W.Workload(name="flat", dims=list(dims), periodic=(1, 1, 1), tau=0.8, kappa=0.3, eps=1.0,
                    E_ext=(0.0, 0.0, 0.0), levels=levels, coarse_sweeps=12)
    psi0 = W.random_fields(dims[0] * dims[1] * dims[2], 5).reshape(dims[::-1])
    out = []
    for lists in (0, 1):
        sim = es.Simulation(wl, precision, overrides=dict(near_list_cells=lists))
        sim.map_particles()
        assert _levels_in_cluster(sim) == (want if lists == 0 else [])
        sim.set_field(es.FIELD_PSI, psi0)
        sim.solve(forced_cycles=2)
        out.append(sim.field(es.FIELD_PSI))
        sim.close()
    if precision == es.ES_FP64:
        assert rel_l2(out[0], out[1]) < 1e-12
    else:
        np.testing.assert_array_equal(out[0], out[1])
