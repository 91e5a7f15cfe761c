"""The forms a step takes by the size of its input: blocks of 64 threads that
load their records ahead (up to 640 particles an SM, 97 280 on 152 SMs), blocks
of 256 above; the one-kernel rebuild and graphs of several steps below that
limit, the chain of kernels above it and under per-kernel timing; and the
persistent kernel's two builds (up to 512 particles an SM, 77 824, and above).

All of them do the same arithmetic per particle in the same order, so every
form gives the same bits.

(Where the lines lie by now: test_builds_asked_for_and_builds_that_come_up.)
"""
import numpy as np
import pytest

from paper_1702_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

FIELDS = ("pos", "vel", "rho", "order", "cell")


@pytest.fixture(scope="module")
def sphmod():
    from paper_1702_07760_gb300 import build as B
    from paper_1702_07760_gb300 import sph
    B.build()
    sph.load()
    return sph


def _same(a, b):
    for f in FIELDS:
        assert np.array_equal(a.read(f), b.read(f)), f
    assert a.list_builds == b.list_builds and a.step_index == b.step_index


# (2-D) one block, both sides of 77 824 (272 x 286 and 273 x 286 particles) and of 97 280
# (311 x 312 and 312 x 312), with oil, walls and list rebuilds; (3-D) both sides of 97 280
@pytest.mark.parametrize("shape", [(1, 2), (266, 280), (267, 280), (305, 306), (306, 306), (39, 40, 40), (40, 40, 40)])
def test_every_form_gives_the_same_bits(sphmod, shape):
    w = WL.drop_tank(len(shape), shape, drop_d_dx=min(shape) / 3, seed=sum(shape), perturb=True)
    dt = WL.stable_dt(w.params)
    graph, eager, timed, persistent = (sphmod.Simulation.from_workload(w) for _ in range(4))
    graph.run(dt, 3)
    graph.run(dt, 11)                  # a graph of eight steps and three of one
    eager.run(dt, 14, graph=False)
    timed.timing(True)
    timed.run(dt, 14)
    timed.timing(False)
    persistent.run_persistent(dt, 14)
    assert graph.list_builds >= 2 or min(shape) < 4
    for s in (eager, timed, persistent):
        _same(graph, s)
    for s in (graph, eager, timed):    # a forced build and the sweeps of stage 0
        s.timing(s is timed)
        s.eval_rates()
        s.timing(False)
    for f in ("acc", "drho", "pressure", "rho_eval", "tensor"):
        a = graph.read(f)
        assert np.array_equal(a, eager.read(f)) and np.array_equal(a, timed.read(f)), f


# both sides of 1 536 particles an SM (233 472 on 152 SMs; 486 x 480 and 487 x 480 particles),
# above which a graph's sweeps start while the sweep before them ends
@pytest.mark.parametrize("shape", [(480, 474), (481, 474)])
def test_overlapped_sweeps_give_the_same_bits(sphmod, shape):
    w = WL.drop_tank(2, shape, drop_d_dx=100, seed=sum(shape), perturb=True)
    dt = WL.stable_dt(w.params)
    graph, eager, timed = (sphmod.Simulation.from_workload(w) for _ in range(3))
    graph.run(dt, 14)
    eager.run(dt, 14, graph=False)
    timed.timing(True)
    timed.run(dt, 14)
    timed.timing(False)
    for s in (eager, timed):
        _same(graph, s)


def test_periodic_and_piston_in_the_small_forms(sphmod):
    w = WL.wave_tank_small()
    m = w.meta["piston"]
    dt = WL.stable_dt(w.params)
    sims = [sphmod.Simulation.from_workload(w) for _ in range(3)]
    for s in sims:
        s.set_piston(m["axis"], m["amp"], m["omega"], m["phase"], m["t_end"])
    sims[0].run(dt, 20)
    sims[1].timing(True)
    sims[1].run(dt, 20)
    sims[2].run_persistent(dt, 20)
    for s in sims[1:]:
        _same(sims[0], s)
        assert s.time == sims[0].time


@pytest.mark.parametrize("block,grid", [(128, 4), (128, 9), (512, 3)])
def test_chunks_beyond_the_warps(sphmod, block, grid):
    """A grid with fewer warps than chunks of 32 particles: the first chunk of each warp is its
    own, the others come from the counter."""
    w = WL.drop_tank(2, (33, 41), drop_d_dx=10, seed=33, perturb=True)
    dt = WL.stable_dt(w.params)
    ref = sphmod.Simulation.from_workload(w)
    ref.run(dt, 12)
    s = sphmod.Simulation.from_workload(w)
    s.set_launch_shape(block, grid, True)
    s.run_persistent(dt, 12)
    _same(ref, s)


# above 1 536 particles an SM (233 472 on 152 SMs): 62 x 66 x 78 = 319 176 particles, 700 x 360 = 252 000
@pytest.mark.parametrize("shape", [(56, 60, 72), (694, 354)])
def test_large_inputs_give_the_same_bits_in_every_form(sphmod, shape):
    """Each sweep starts after the one before it has ended, whose records it reads through the
    read-only path; steps, and rates on a fresh list."""
    w = WL.drop_tank(len(shape), shape, drop_d_dx=min(shape) / 3, seed=sum(shape), perturb=True)
    dt = WL.stable_dt(w.params)
    graph, eager, timed, persistent = (sphmod.Simulation.from_workload(w) for _ in range(4))
    graph.run(dt, 9)
    eager.run(dt, 9, graph=False)
    timed.timing(True)
    timed.run(dt, 9)
    timed.timing(False)
    persistent.run_persistent(dt, 9)
    for s in (eager, timed, persistent):
        _same(graph, s)
    for s in (graph, timed):
        s.timing(s is timed)
        s.eval_rates()
        s.timing(False)
    for f in ("acc", "drho", "pressure", "rho_eval", "tensor"):
        assert np.array_equal(graph.read(f), timed.read(f)), f


# The lines as they stand, in particles an SM (x 152 SMs): blocks that load ahead up to 384 in
# 2-D (58 368; 208 x 280 = 58 240 and 209 x 280 = 58 520 particles) and 768 in 3-D (116 736; 36 x 54 x 60 =
# 116 640 and 37 x 54 x 60 = 119 880); a certain build in one kernel up to 512 (77 824; 272 x 286 and
# 273 x 286), a step's up to 1 536 (233 472; 48 x 64 x 76 = 233 472 and 49 x 64 x 76 = 238 336).
@pytest.mark.parametrize("shape", [(202, 274), (203, 274), (266, 280), (267, 280),
                                   (30, 48, 54), (31, 48, 54), (42, 58, 70), (43, 58, 70)])
def test_builds_asked_for_and_builds_that_come_up(sphmod, shape):
    """Builds that the host asks for (a first run, a new state, a new step size, a forced build)
    between builds that a step finds due, through every form: the same bits and as many builds."""
    import torch
    w = WL.drop_tank(len(shape), shape, drop_d_dx=min(shape) / 3, seed=sum(shape), perturb=True)
    dt = WL.stable_dt(w.params)
    state = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (w.x, w.u, w.rho)]

    def go(s, run):
        run(s, dt, 9)
        s.load_snapshot(*[a.data_ptr() for a in state])
        run(s, dt, 1)
        run(s, dt, 10)
        run(s, 0.9 * dt, 3)
        s.build_cells()
        run(s, 0.9 * dt, 8)
        s.eval_rates()
        run(s, 0.9 * dt, 2)
        s.set_state(w.x, w.u, w.rho)
        run(s, 0.9 * dt, 2)
        return s

    new = lambda: sphmod.Simulation.from_workload(w)  # noqa: E731
    graph = go(new(), lambda s, d, k: s.run(d, k))
    _same(graph, go(new(), lambda s, d, k: s.run(d, k, graph=False)))
    _same(graph, go(new(), lambda s, d, k: s.run_persistent(d, k)))
    timed = new()
    timed.timing(True)
    _same(graph, go(timed, lambda s, d, k: s.run(d, k)))


@pytest.mark.parametrize("every", [1, 3, 8])
@pytest.mark.parametrize("shape", [(40, 40), (300, 300)])
def test_fixed_cadences(sphmod, shape, every):
    """Every, every third and every eighth step builds, below and above 512 particles an SM."""
    w = WL.drop_tank(2, shape, drop_d_dx=min(shape) / 3, seed=every, perturb=True)
    w.params["rebuild_every"] = every
    dt = 0.25 * WL.stable_dt(w.params)   # a fixed cadence reports a motion beyond the skin
    graph, eager, persistent = (sphmod.Simulation.from_workload(w) for _ in range(3))
    graph.run(dt, 3)
    graph.run(dt, 17)
    eager.run(dt, 20, graph=False)
    persistent.run_persistent(dt, 20)
    assert graph.list_builds >= 20 // every
    for s in (eager, persistent):
        _same(graph, s)
