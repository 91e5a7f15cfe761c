"""FP64 diagnostics over tiles of 1 024 particles: sizes around whole tiles, one
simulation and uneven batches, against the oracle.

Every quantity is a sum of n FP64 terms in some order, so two orders differ by
at most n eps times the sum of the terms' magnitudes: n <= 1e4 here, and the
bound used is 1e-12 of that sum.
"""
import numpy as np
import pytest

import oracle
from paper_1702_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

EPS = 1e-12


@pytest.fixture(scope="module")
def sphmod():
    from paper_1702_07760_gb300 import build as B
    from paper_1702_07760_gb300 import sph
    B.build()
    sph.load()
    return sph


def _check(d, w):
    r = oracle.diagnostics(w.params, w.x, w.u, w.phase, w.wall)
    fl = w.wall == 0
    m = np.asarray(w.params["mass"])[w.phase][fl]
    assert abs(d["mass"] - r["mass"]) <= EPS * r["mass"]
    assert np.abs(d["momentum"] - r["momentum"]).max() <= EPS * (m[:, None] * np.abs(w.u[fl])).sum()
    assert abs(d["e_kin"] - r["e_kin"]) <= EPS * max(r["e_kin"], 1e-300)
    g = np.abs(np.asarray(w.params["g"][:w.dim]))
    assert abs(d["e_pot"] - r["e_pot"]) <= EPS * (m * (np.abs(w.x[fl]) @ g)).sum()
    assert d["u_max"] == np.sqrt((w.u[fl] ** 2).sum(1)).max() or abs(d["u_max"] / r["u_max"] - 1) < 1e-15
    assert d["n_oil"] == int(((w.phase == 1) & fl).sum())
    if d["n_oil"]:
        assert np.abs(d["centroid"] - r["centroid"]).max() <= EPS * np.abs(w.x[fl]).max()
        assert abs(d["sphericity"] - r["sphericity"]) < 1e-9


# 1 023, 1 024, 1 025 and 4 097 fluid particles without walls, and closed tanks
@pytest.mark.parametrize("n", [1, 255, 1023, 1024, 1025, 4097])
def test_particle_counts_around_a_tile(sphmod, n):
    w = WL.drop_tank(2, (64, 72), drop_d_dx=20, seed=n, perturb=True, wall_layers=3)
    keep = np.flatnonzero(w.wall == 0)[:n]
    w = WL.Workload(w.name, w.params, w.x[keep], w.u[keep], w.rho[keep], w.phase[keep], w.wall[keep], w.meta)
    sim = sphmod.Simulation.from_workload(w)
    _check(sim.diagnostics(), w)
    sim.build_cells()
    _check(sim.diagnostics(), w)   # the same through a sorted state


def test_three_dimensions_and_an_uneven_batch(sphmod):
    w = WL.drop_tank(3, (11, 13, 17), drop_d_dx=7, seed=3, perturb=True)
    sim = sphmod.Simulation.from_workload(w)
    sim.build_cells()
    for _ in range(2):
        _check(sim.diagnostics(), w)
    ws = WL.drop_batch_2d(k=5, seed=78, d_range=(5.0, 14.0), perturb=True)
    sim = sphmod.Simulation.batch(ws)
    sim.build_cells()
    for _ in range(2):
        for d, q in zip(sim.diagnostics_instances(), ws):
            _check(d, q)


def _state_of(sim, w):
    return WL.Workload(w.name, w.params, sim.read("pos"), sim.read("vel"), sim.read("rho"), w.phase, w.wall, w.meta)


def test_periodic_tank_with_a_piston(sphmod):
    """Positions wrapped into the box and prescribed velocities, after steps and before the first."""
    w = WL.wave_tank_small()
    m = w.meta["piston"]
    sim = sphmod.Simulation.from_workload(w)
    sim.set_piston(m["axis"], m["amp"], m["omega"], m["phase"], m["t_end"])
    _check(sim.diagnostics(), _state_of(sim, w))
    sim.run(WL.stable_dt(w.params), 12)
    _check(sim.diagnostics(), _state_of(sim, w))


def test_instances_without_oil_among_others(sphmod):
    ws = WL.drop_batch_2d(k=5, seed=79, d_range=(5.0, 14.0), perturb=True)
    for q in (0, 3):
        ws[q].phase[:] = 0
    sim = sphmod.Simulation.batch(ws)
    for _ in range(2):
        for q, (d, w) in enumerate(zip(sim.diagnostics_instances(), ws)):
            _check(d, w)
            assert (d["n_oil"] == 0) == (q in (0, 3))
            if q in (0, 3):
                assert not np.any(d["centroid"])
        sim.build_cells()


@pytest.mark.parametrize("bad", ["nan", "-nan", "inf", "-inf"])
def test_velocities_that_are_not_finite(sphmod, bad):
    """The largest speed leaves out a NaN and keeps an infinity; sums over it are not finite, and
    what does not read velocities is as it was."""
    v = {"nan": np.nan, "-nan": -np.nan, "inf": np.inf, "-inf": -np.inf}[bad]
    w = WL.drop_tank(2, (40, 44), drop_d_dx=12, seed=80, perturb=True)
    at = np.flatnonzero(w.wall == 0)[717]
    u = w.u.copy()
    u[at, 1] = v
    sim = sphmod.Simulation.from_workload(w)
    ref = sim.diagnostics()
    sim.set_state(w.x, u, w.rho)
    d = sim.diagnostics()
    others = np.delete(w.u, at, 0)[np.delete(w.wall, at) == 0]
    if np.isnan(v):
        assert d["u_max"] == np.sqrt((others ** 2).sum(1).max()) or \
            abs(d["u_max"] / np.sqrt((others ** 2).sum(1).max()) - 1) < 1e-15
        assert np.isnan(d["e_kin"]) and np.isnan(d["momentum"][1])
    else:
        assert d["u_max"] == np.inf and d["e_kin"] == np.inf and d["momentum"][1] == v
    for k in ("mass", "e_pot", "sphericity", "n_oil"):
        assert d[k] == ref[k], k
    assert d["momentum"][0] == ref["momentum"][0] and np.array_equal(d["centroid"], ref["centroid"])
