"""The local correction at a solve's start: clusters solved in shared memory
(one flip, flips close together) and in global memory (boxes too large, or
longer than a periodic axis), against a start without it."""
import numpy as np
import pytest

import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _spheres(dims, periodic, x, levels):
    n = len(x)
    wl = W.Workload(name="local", dims=dims, periodic=periodic, tau=1.0, kappa=0.3, eps=1.0, E_ext=(1e-3, 0.0, 0.0),
                    levels=levels, res_rf=1e-8, coarse_sweeps=16, max_cycles=200)
    return W._set_particles(wl, np.array(x, dtype=float), np.full(n, 4.2), np.array([i % 2 for i in range(n)]),
                            np.ones(n), np.full(n, 1.3))


@pytest.mark.parametrize("dims,periodic,x,levels", [
    ((64, 64, 64), (1, 1, 1), [(31.37, 32.11, 30.83)], 3),
    ((64, 64, 64), (1, 1, 1), [(1.37, 62.11, 0.83)], 3),                         # across the periodic faces
    ((64, 48, 56), (1, 0, 0), [(31.37, 6.11, 50.2)], 3),                         # against walls
    ((64, 64, 64), (1, 1, 1), [(20.37, 32.11, 30.83), (34.1, 30.7, 33.9)], 3),   # a chain of flips
    ((16, 48, 48), (1, 1, 1), [(7.37, 24.11, 22.83)], 2),                        # the box exceeds the x axis
])
def test_local_correction(dims, periodic, x, levels):
    """Both solves end below 1e-8 of the first residual, so the potentials
    differ by at most 2e-8 cond(A) < 2e-8 (12 + kappa^2) / kappa^2 = 2.7e-6."""
    wl = _spheres(dims, periodic, x, levels)
    sims = [es.Simulation(wl, es.ES_MIXED32, overrides=dict(fast_update_cells=f)) for f in (1, 2 ** 31 - 1)]
    for s in sims:
        s.map_particles()
        s.solve()
    own = sims[0].field(es.FIELD_OWNER)
    rng = np.random.Generator(np.random.PCG64(3))
    flipped = 0
    for _ in range(6):
        wl.x = wl.x + rng.uniform(-0.04, 0.04, wl.x.shape)
        info = []
        for s in sims:
            s.set_particles(wl.x, wl.v, wl.w)
            s.map_particles()
            info.append(s.solve())
        new = sims[0].field(es.FIELD_OWNER)
        now = int(((new >= 0) != (own >= 0)).sum())
        flipped += now
        own = new
        np.testing.assert_array_equal(own, sims[1].field(es.FIELD_OWNER))
        a, b = (s.field(es.FIELD_PSI) for s in sims)
        assert np.linalg.norm(a - b) <= 2.7e-6 * np.linalg.norm(b)
        if now:  # (else each solve starts from its own last residual)
            assert info[0]["r0"] <= info[1]["r0"] * (1 + 1e-3)
    assert flipped > 0
    for s in sims:
        s.close()


CLUSTERS = [  # solved in shared memory; and, on a short axis, from the list in global memory
    ((64, 64, 64), (1, 1, 1), [(31.37, 32.11, 30.83)], 3),
    ((16, 48, 48), (1, 1, 1), [(7.37, 24.11, 22.83)], 2),
]


def _moves(wl, sims, n):
    """The solves' records of n small moves of the spheres; True where a cell flipped."""
    rng = np.random.Generator(np.random.PCG64(3))
    for s in sims:
        s.map_particles()
        s.solve()
    own = sims[0].field(es.FIELD_OWNER)
    for _ in range(n):
        wl.x = wl.x + rng.uniform(-0.04, 0.04, wl.x.shape)
        info = []
        for s in sims:
            s.set_particles(wl.x, wl.v, wl.w)
            s.map_particles()
            info.append(s.solve())
        new = sims[0].field(es.FIELD_OWNER)
        yield bool(((new >= 0) != (own >= 0)).any()), info
        own = new


@pytest.mark.parametrize("dims,periodic,x,levels", CLUSTERS)
def test_scaled_problem_gives_scaled_bits(dims, periodic, x, levels):
    """The solve is linear and its sums hold their range: surface potentials and
    charges times 2^-40 give the potential times 2^-40 to the last bit (the
    squares of the residuals, below 1e-45 then, are out of FP32's range)."""
    wl = [_spheres(dims, periodic, x, levels) for _ in range(2)]
    wl[1].zeta, wl[1].q = wl[1].zeta * 2.0 ** -40, wl[1].q * 2.0 ** -40
    sims = [es.Simulation(w, es.ES_MIXED32, overrides=dict(fast_update_cells=1)) for w in wl]
    flips = 0
    for flipped, info in _moves(wl[0], sims, 6):
        flips += flipped
        assert info[0]["cycles"] == info[1]["cycles"]
        np.testing.assert_array_equal(sims[1].field(es.FIELD_PSI) * 2.0 ** 40, sims[0].field(es.FIELD_PSI))
    assert flips > 0
    for s in sims:
        s.close()


@pytest.mark.parametrize("dims,periodic,x,levels", CLUSTERS)
def test_reported_residual_after_the_correction(dims, periodic, x, levels):
    """The first residual of a solve that corrects locally, kept by the change of
    r^2 over the clusters, against the residual of its potential formed in full:
    within the 1 % of the tolerance that the carried residual may drift by.  At a
    tolerance of 1e-3 of the first solve's residual (a flip leaves some 3e-2)
    the correction does without V-cycles, and a start without it needs them."""
    wl = _spheres(dims, periodic, x, levels)
    wl.res_rf = 1e-3
    sims = [es.Simulation(wl, es.ES_MIXED32, overrides=dict(fast_update_cells=f)) for f in (1, 2 ** 31 - 1)]
    spared = 0
    for flipped, info in _moves(wl, sims, 6):
        if flipped and info[0]["cycles"] == 0:
            full = sims[0].solve(forced_cycles=0)["r0"]
            assert abs(full - info[0]["r0"]) <= 0.01 * info[0]["tol"]
            spared += info[1]["cycles"] > 0
    assert spared > 0
    for s in sims:
        s.close()


@pytest.mark.parametrize("precision,dims", [(es.ES_MIXED32, (96, 96, 96)), (es.ES_MIXED32, (84, 84, 84)),
                                            (es.ES_FP64, (64, 64, 64))])
def test_many_mappings_between_solves(precision, dims):
    """Spheres mapped to and fro until more cells have flipped than the list of
    flipped cells holds (2^16): the next solve ends where one does whose
    context was mapped there once, both below 1e-10 of the first residual, so
    within 2e-10 (12 + kappa^2) / kappa^2 = 2.7e-8.  (84: not colour-split,
    FP64: neither keeps a list.)"""
    wl = W.mixed_box(dims=dims, periodic=(1, 1, 1), levels=2, n_spheres=60 if dims[0] > 64 else 20, radius=4.2)
    wl.v[:] = 0.0
    wl.w[:] = 0.0
    x0 = wl.x.copy()
    sims = [es.Simulation(wl, precision, overrides=dict(fast_update_cells=1)) for _ in range(2)]
    for s in sims:
        s.map_particles()
        s.solve(forced_cycles=3)
    own = sims[0].field(es.FIELD_OWNER) >= 0
    flips = 0
    for k in range(1, 61):
        sims[0].set_particles(x0 + (0.4 if k % 2 else 0.0), wl.v, wl.w)
        sims[0].map_particles()
        if k in (1, 2):
            new = sims[0].field(es.FIELD_OWNER) >= 0
            flips += 30 * int((new != own).sum())
            own = new
    assert flips > (1 << 16) or precision == es.ES_FP64
    for s in sims:
        s.set_particles(x0 + 0.1, wl.v, wl.w)
        s.map_particles()
        s.solve()
    np.testing.assert_array_equal(sims[0].field(es.FIELD_OWNER), sims[1].field(es.FIELD_OWNER))
    a, b = (s.field(es.FIELD_PSI) for s in sims)
    assert np.linalg.norm(a - b) <= 2.7e-8 * np.linalg.norm(b)
    for s in sims:
        s.close()
