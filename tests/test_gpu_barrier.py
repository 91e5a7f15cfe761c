"""A grid barrier that gives up, in every call that can meet one: the wait is
bounded (one second, whatever is queued behind it), the call that waits for the
stream reports it, nothing is integrated or learned on unfinished lists, and the
handle goes on from the state it had, without being given one.

The barrier is put in a state that no arrival completes (test support of the
library), so the launches wait out their limit and return; nothing faults.
"""
import time

import numpy as np
import pytest

from paper_1702_07760_gb300 import workloads as WL
from test_gpu_surrogate import _case, env  # noqa: F401

pytestmark = pytest.mark.gpu

FIELDS = ("pos", "vel", "rho", "order", "cell")


def _tank(dim):
    return WL.drop_tank(2, (60, 66), drop_d_dx=20, seed=7, perturb=True) if dim == 2 else \
        WL.drop_tank(3, (14, 13, 15), drop_d_dx=7, seed=8, perturb=True)


def _times_out(sph, f):
    t = time.perf_counter()
    with pytest.raises(sph.SphError) as e:
        f()
    assert e.value.code == -8
    # one wait of a second; a second one would be past this
    assert time.perf_counter() - t < 1.9


def _same(a, b, fields=FIELDS):
    for f in fields:
        assert np.array_equal(a.read(f), b.read(f)), f
    assert a.step_index == b.step_index


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", ["graph", "eager", "persistent"])
def test_a_run_goes_on_after_a_time_out(env, dim, form):  # noqa: F811
    _, sph = env
    w = _tank(dim)
    dt = WL.stable_dt(w.params)
    s, ref = (sph.Simulation.from_workload(w) for _ in range(2))
    s.run(dt, 1)                       # the kernels are loaded before the wait is timed
    s.run_persistent(dt, 1)
    ref.run(dt, 2)

    def run(h, d, k):
        if form == "persistent":
            h.run_persistent(d, k)
        else:
            h.run(d, k, graph=form == "graph")

    # a new step size builds the lists: 19 steps are two graphs of eight and three of one
    run(s, 0.9 * dt, 19)
    run(ref, 0.9 * dt, 19)
    _same(s, ref)
    s.test_stall_barrier()
    _times_out(sph, lambda: run(s, 0.8 * dt, 19))
    _same(s, ref)                      # no step was made, and none is counted
    run(s, 0.8 * dt, 19)
    run(ref, 0.8 * dt, 19)
    _same(s, ref)
    assert s.time == ref.time


@pytest.mark.parametrize("shape", [(128, 4), (512, 1)])
def test_launch_shapes_smaller_than_the_rebuild(env, shape):  # noqa: F811
    """The stalled state holds for the rebuild's grid too, whatever the persistent one's."""
    _, sph = env
    w = _tank(2)
    dt = WL.stable_dt(w.params)
    s, ref = (sph.Simulation.from_workload(w) for _ in range(2))
    s.eval_rates()
    s.sync()
    s.set_launch_shape(*shape)
    s.test_stall_barrier()
    _times_out(sph, lambda: s.run(dt, 3))
    s.run(dt, 3)
    ref.run(dt, 3)
    _same(s, ref)


def test_before_the_first_build(env):  # noqa: F811
    """Nothing is there yet: empty lists, then a state given, then the first build."""
    _, sph = env
    w = _tank(3)
    dt = WL.stable_dt(w.params)
    s, ref = (sph.Simulation.from_workload(w) for _ in range(2))
    s.test_stall_barrier()
    with pytest.raises(sph.SphError) as e:
        s.run(dt, 9)
    assert e.value.code == -8 and s.step_index == 0 and s.list_builds == 0
    s.set_state(w.x, w.u, w.rho)
    s.run(dt, 9)
    ref.run(dt, 9)
    _same(s, ref)


def test_rates_and_queries(env):  # noqa: F811
    _, sph = env
    w = _tank(2)
    s, ref = (sph.Simulation.from_workload(w) for _ in range(2))
    ref.eval_rates()
    s.eval_rates()
    s.sync()
    for query in (lambda: (s.eval_rates(), s.sync()), lambda: (s.step(WL.stable_dt(w.params)), s.sync()),
                  lambda: (s.build_cells(), s.sync()), s.neighbours, s.pair_stats):
        s.test_stall_barrier()
        _times_out(sph, query)
    s.eval_rates()
    _same(s, ref, FIELDS + ("acc", "drho", "pressure", "rho_eval", "tensor"))


@pytest.mark.parametrize("dim", [2, 3])
def test_the_network_keeps_its_weights(env, dim):  # noqa: F811
    torch, sph = env
    w, norm, flat = _case(dim, 70 + dim)
    rng = np.random.Generator(np.random.PCG64(71))
    free = (w.wall == 0)[:, None]
    t = [torch.tensor(a, dtype=torch.float64, device="cuda")
         for a in (w.x + free * rng.normal(0, 1e-6, w.x.shape), w.u + free * rng.normal(0, 1e-2, w.u.shape),
                   w.rho * (1 + rng.normal(0, 1e-4, w.n)))]
    s, ref = (sph.Simulation.from_workload(w) for _ in range(2))
    for h in (s, ref):
        h.surrogate_init(flat, norm)
        h.surrogate_train_step(*[a.data_ptr() for a in t], update=False)
    for _ in range(2):                 # the launched step, then the replayed one
        before = s.surrogate_weights()
        s.test_stall_barrier()
        _times_out(sph, lambda: s.surrogate_train_step(*[a.data_ptr() for a in t], lr=1e-3))
        assert np.array_equal(s.surrogate_weights(), before)
        s.surrogate_train_step(*[a.data_ptr() for a in t], lr=1e-3)
        _, g = ref.surrogate_train_step(*[a.data_ptr() for a in t], lr=1e-3, want_grad=True)
        big = np.abs(g) > 1e-3 * np.abs(g).max()
        # the same count of updates: Adam's step is lr times a ratio that the gradient's
        # rounding (1e-5 of its norm) moves little where the gradient is not small
        assert np.abs(s.surrogate_weights() - ref.surrogate_weights())[big].max() < 2e-2 * 1e-3
    s.test_stall_barrier()
    _times_out(sph, lambda: (s.surrogate_advance(8), s.sync()))
    _same(s, ref, ("pos", "vel", "rho"))
    s.surrogate_advance(8)
    s.sync()
    assert s.step_index == 8
