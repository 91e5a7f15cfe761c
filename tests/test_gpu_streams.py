"""Handles on streams of the caller's that are not ordinary ones: of a green context, which
gives its kernels a part of the multiprocessors, and the legacy default stream, which cannot be
captured into a graph."""
import ctypes as C

import numpy as np
import pytest

from paper_1702_07760_gb300 import workloads as WL
from test_gpu_surrogate import _case, env  # noqa: F401

pytestmark = pytest.mark.gpu


class _Resource(C.Structure):
    _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sm_count", C.c_uint), ("rest", C.c_ubyte * 44)]


@pytest.fixture
def green_stream(env):  # noqa: F811
    """A stream of a green context of 16 multiprocessors or a few more."""
    torch, _ = env
    torch.zeros(1, device="cuda")        # the primary context
    L = C.CDLL("libcuda.so.1")
    if not hasattr(L, "cuGreenCtxStreamCreate"):
        pytest.skip("no green contexts in this driver")
    dev, group, left = C.c_int(), _Resource(), _Resource()
    all_sms = _Resource()
    count = C.c_uint(1)
    desc, ctx, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()

    def ok(r):
        if r:
            pytest.skip(f"no green context here (driver error {r})")

    ok(L.cuDeviceGet(C.byref(dev), torch.cuda.current_device()))
    ok(L.cuDeviceGetDevResource(dev, C.byref(all_sms), 1))
    ok(L.cuDevSmResourceSplitByCount(C.byref(group), C.byref(count), C.byref(all_sms), C.byref(left), 0, 16))
    ok(L.cuDevResourceGenerateDesc(C.byref(desc), C.byref(group), 1))
    ok(L.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1))
    ok(L.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0))
    yield stream.value, group.sm_count, all_sms.sm_count
    L.cuStreamSynchronize(stream)
    L.cuStreamDestroy_v2(stream)
    L.cuGreenCtxDestroy(ctx)


# 16 multiprocessors hold 32 blocks of the cooperative rebuild at once, the whole device 304: 4 752
# particles ask for 19 blocks, 23 760 for 93, 103 776 (above 1 536 on each of 16) for none
@pytest.mark.parametrize("shape", [(60, 66), (129, 170), (270, 370), (14, 13, 15)])
def test_part_of_the_multiprocessors(env, green_stream, shape):  # noqa: F811
    torch, sph = env
    stream, sms, all_sms = green_stream
    assert 0 < sms < all_sms
    w = WL.drop_tank(len(shape), shape, drop_d_dx=min(shape) / 3, seed=sum(shape), perturb=True)
    dt = WL.stable_dt(w.params)
    state = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (w.x, w.u, w.rho)]
    torch.cuda.synchronize()
    s, ref = sph.Simulation.from_workload(w, stream=stream), sph.Simulation.from_workload(w)
    # graphs with a conditional node (the large form) cannot be instantiated for such a stream
    graph = w.n <= 1536 * sms
    for h in (s, ref):
        h.run(dt, 11, graph=graph)
        h.run(0.9 * dt, 3, graph=False)
        h.eval_rates()
        h.run(0.9 * dt, 2, graph=graph)
        h.load_snapshot(*[a.data_ptr() for a in state])
        h.run(0.9 * dt, 3, graph=graph)
    for f in ("pos", "vel", "rho", "order", "cell"):
        assert np.array_equal(s.read(f), ref.read(f)), f
    assert s.list_builds == ref.list_builds
    s.close()
    ref.close()


@pytest.mark.parametrize("stream", [1, 2])   # cudaStreamLegacy, cudaStreamPerThread
@pytest.mark.parametrize("dim", [2, 3])
def test_training_on_default_streams(env, dim, stream):  # noqa: F811
    """Every step after the first replays a graph where the stream can be captured, and is
    launched where it cannot: the loss to the order of FP64 sums (1e-10), the gradient to that of
    FP32 ones (1e-5 of its norm)."""
    torch, sph = env
    w, norm, flat = _case(dim, 50 + dim)
    rng = np.random.Generator(np.random.PCG64(51))
    free = (w.wall == 0)[:, None]
    t = [torch.tensor(a, dtype=torch.float64, device="cuda")
         for a in (w.x + free * rng.normal(0, 1e-6, w.x.shape), w.u + free * rng.normal(0, 1e-2, w.u.shape),
                   w.rho * (1 + rng.normal(0, 1e-4, w.n)))]
    torch.cuda.synchronize()
    s, ref = sph.Simulation.from_workload(w, stream=stream), sph.Simulation.from_workload(w)
    for h in (s, ref):
        h.surrogate_init(flat, norm)
    for _ in range(3):
        s.surrogate_train_step(*[a.data_ptr() for a in t], lr=1e-3)
    assert np.abs(s.surrogate_weights() - flat).max() > 1e-3   # three updates were made
    s.surrogate_init(flat, norm)
    for _ in range(3):
        loss, g = s.surrogate_train_step(*[a.data_ptr() for a in t], update=False, want_grad=True)
        loss1, g1 = ref.surrogate_train_step(*[a.data_ptr() for a in t], update=False, want_grad=True)
        assert abs(loss - loss1) <= 1e-10 * loss1
        assert np.linalg.norm(g - g1) <= 1e-5 * np.linalg.norm(g1)


def test_handles_side_by_side(env):  # noqa: F811
    """Several handles, each on its own stream and thread, whose cooperative rebuilds ask for the
    whole device at the same time (75 k particles: 294 blocks of the 304 it holds), beside training
    steps with streams of their own and a persistent run: the bits of each alone, and no time-out."""
    import threading
    torch, sph = env
    tanks = [WL.drop_tank(2, (250, 288), drop_d_dx=70, seed=1, perturb=True),
             WL.drop_tank(3, (34, 36, 40), drop_d_dx=10, seed=2, perturb=True),
             WL.drop_tank(2, (120, 140), drop_d_dx=30, seed=3, perturb=True),
             WL.drop_tank(2, (350, 380), drop_d_dx=80, seed=4, perturb=True)]

    def steps(s, w, form):
        dt = WL.stable_dt(w.params)
        for k in range(40):
            if form == "persistent":
                s.run_persistent(dt, 10)
            else:
                s.run((1 - 0.01 * (k % 3)) * dt, 10, graph=form == "graph")
            s.eval_rates()
        return [s.read(f) for f in ("pos", "vel", "rho", "order", "acc")]

    w, norm, flat = _case(2, 56)
    t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (w.x, w.u, w.rho)]
    torch.cuda.synchronize()

    def training(s):
        s.surrogate_init(flat, norm)
        return [s.surrogate_train_step(*[a.data_ptr() for a in t], update=False)[0] for _ in range(150)]

    jobs = [(v, f) for v in tanks for f in ("graph", "eager")] + [(tanks[0], "persistent"), (tanks[2], "persistent")]
    alone = [steps(sph.Simulation.from_workload(v), v, f) for v, f in jobs]
    loss = training(sph.Simulation.from_workload(w))
    sims = [sph.Simulation.from_workload(v) for v, _ in jobs]
    trainer = sph.Simulation.from_workload(w)
    got, failed = [None] * len(jobs), []

    def work(q):
        try:
            if q < len(jobs):
                got[q] = steps(sims[q], *jobs[q])
            else:
                assert np.allclose(training(trainer), loss, rtol=1e-10, atol=0)
        except BaseException as e:  # noqa: BLE001 (reported below)
            failed.append((q, e))

    threads = [threading.Thread(target=work, args=(q,)) for q in range(len(jobs) + 1)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
    for a, b in zip(alone, got):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
