"""Training steps after the first replay one captured sequence of launches: a
replayed step equals the same step launched kernel by kernel, whatever state,
targets, step size and network it is given.

Both run the same kernels, so the loss differs by the order of FP64 atomics
only (1e-10 allowed) and the gradient by the order of FP32 ones: a weight
gradient is a sum over nodes in FP32, at most a few hundred roundings of 2^-24
in another order, 1e-5 of the gradient's norm with room for cancellation.
Adam's update is compared with the oracle's from the step's own gradients, where
these are not lost in rounding (as the first step is in test_gpu_surrogate.py).
"""
import numpy as np
import pytest

from oracle import mpnn as O
from test_gpu_surrogate import _case, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _targets(torch, w, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    free = (w.wall == 0)[:, None]
    a = (w.x + free * rng.normal(0, 1e-6, w.x.shape), w.u + free * rng.normal(0, 1e-2, w.u.shape),
         w.rho * (1 + rng.normal(0, 1e-4, w.n)))
    return [torch.tensor(q, dtype=torch.float64, device="cuda") for q in a]


def _state(w, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    free = (w.wall == 0)[:, None]
    return w.x.copy(), w.u + free * rng.normal(0, 1e-2, w.u.shape), w.rho * (1 + rng.normal(0, 1e-5, w.n))


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("timing", [False, True])
def test_replayed_gradients_match_launched_ones(env, dim, timing):  # noqa: F811
    torch, sph = env
    w, norm, flat = _case(dim, 80 + dim)
    sim = sph.Simulation.from_workload(w)
    sim.surrogate_init(flat, norm)
    for k in range(4):
        if k == 3:   # another network and another normalisation
            norm, flat = norm.copy(), flat * 0.9
            norm[-4] *= 1.25
            sim.surrogate_init(flat, norm)
        if timing:
            sim.timing(k == 2)
        s, t = _state(w, 90 + k), _targets(torch, w, 95 + k)
        sim.set_state(*s)
        loss, g = sim.surrogate_train_step(*(q.data_ptr() for q in t), update=False, want_grad=True)
        dt = sim.suggest_dt()
        one = sph.Simulation.from_workload(w)
        one.surrogate_init(flat, norm)
        one.set_state(*s)
        loss1, g1 = one.surrogate_train_step(*(q.data_ptr() for q in t), update=False, want_grad=True)
        assert abs(loss - loss1) <= 1e-10 * loss1
        assert np.linalg.norm(g - g1) <= 1e-5 * np.linalg.norm(g1)
        assert dt == one.suggest_dt()


def test_replayed_updates_take_their_own_step_size(env):  # noqa: F811
    torch, sph = env
    w, norm, flat = _case(2, 85)
    sim = sph.Simulation.from_workload(w)
    sim.surrogate_init(flat, norm)
    m = v = np.zeros_like(flat)
    for k, lr in enumerate((1e-3, 3e-4, 1e-2, 1e-3)):
        t = _targets(torch, w, 100 + k)
        theta = sim.surrogate_weights()
        _, g = sim.surrogate_train_step(*(q.data_ptr() for q in t), lr=lr, update=True, want_grad=True)
        expect, m, v = O.adam(theta, g, m, v, k + 1, lr)
        big = np.abs(g) > 1e-4 * np.abs(g).max()
        assert np.abs(sim.surrogate_weights() - expect)[big].max() < 2e-3 * lr


@pytest.mark.parametrize("dim", [2, 3])
def test_replays_between_steps_and_builds(env, dim):  # noqa: F811
    """What moves the state, the lists and the handle's forms between two training steps: each
    replay against the first step of a handle that has come the same way (a rates evaluation in
    the place of each training step before, which builds the same lists)."""
    from paper_1702_07760_gb300 import workloads as WL
    torch, sph = env
    w, norm, flat = _case(dim, 88 + dim)
    dt = WL.stable_dt(w.params)

    def timed(s):
        s.timing(True)
        s.run(dt, 3)
        s.timing(False)

    ways = [lambda s: None, lambda s: s.run(dt, 5), lambda s: s.run_persistent(dt, 3), lambda s: s.build_cells(),
            lambda s: s.run(0.9 * dt, 9), timed, lambda s: s.set_state(*_state(w, 89)),
            lambda s: (s.set_dt_scales([0.5]), s.run(dt, 2)), lambda s: s.set_launch_shape(128, 4)]
    sim = sph.Simulation.from_workload(w)
    sim.surrogate_init(flat, norm)
    for k, way in enumerate(ways):
        way(sim)
        targets = _targets(torch, w, 110 + k)
        t = [q.data_ptr() for q in targets]
        loss, g = sim.surrogate_train_step(*t, update=False, want_grad=True)
        one = sph.Simulation.from_workload(w)
        for before in ways[:k]:
            before(one)
            one.eval_rates()
        way(one)
        one.surrogate_init(flat, norm)
        loss1, g1 = one.surrogate_train_step(*t, update=False, want_grad=True)
        assert abs(loss - loss1) <= 1e-10 * loss1, k
        assert np.linalg.norm(g - g1) <= 1e-5 * np.linalg.norm(g1), k
        for f in ("pos", "vel", "rho", "order"):
            assert np.array_equal(sim.read(f), one.read(f)), (k, f)
        one.close()
