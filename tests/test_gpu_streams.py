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
