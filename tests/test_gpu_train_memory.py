"""The backward pass with one set of buffers for all layers, on one stream: taken where a set a
layer does not fit the device's memory (and beyond 2^20 particles).  The same kernels on the same
values, so the loss agrees to the order of FP64 sums (1e-10) and the gradient to that of FP32 ones
(1e-5 of its norm; a few hundred roundings of 2^-24 a weight).
"""
import numpy as np
import pytest

from paper_1702_07760_gb300 import surrogate_layout as SL
from paper_1702_07760_gb300 import workloads as WL
from test_gpu_surrogate import env  # noqa: F401

pytestmark = pytest.mark.gpu

GB = 1 << 30


def _norm(w):
    dim, c0 = w.dim, w.params["c0"]
    return SL.make_norm(dim, np.zeros(2 * dim + 4),
                        np.concatenate([np.full(dim, 0.006 * c0), [1e-3], [1, 1], np.full(dim, 0.05), [1e-3]]),
                        np.zeros(2 * dim + 1), np.concatenate([np.full(dim, 1e-6), np.full(dim, 1e-2), [1e-4]]),
                        20.0, 8 * WL.stable_dt(w.params), 0.008 * c0, 1.5e-3)


@pytest.mark.parametrize("stepped", [False, True])
def test_one_set_of_buffers_where_memory_is_short(env, stepped):  # noqa: F811
    torch, sph = env
    # 506 x 516 = 261 096 particles: a set a layer is 10 080 bytes a particle (2.45 GB), one set 4 192 (1.02 GB)
    w = WL.drop_tank(2, (500, 510), drop_d_dx=120, seed=5, perturb=True)
    norm, flat = _norm(w), SL.init_weights(2, seed=6, out_scale=1.0)
    rng = np.random.Generator(np.random.PCG64(7))
    free = (w.wall == 0)[:, None]
    t = [torch.tensor(a, dtype=torch.float64, device="cuda")
         for a in (w.x + free * rng.normal(0, 1e-6, w.x.shape), w.u + free * rng.normal(0, 1e-2, w.u.shape),
                   w.rho * (1 + rng.normal(0, 1e-4, w.n)))]
    p = [a.data_ptr() for a in t]
    ref, s = (sph.Simulation.from_workload(w) for _ in range(2))
    for h in (ref, s):
        h.surrogate_init(flat, norm)
    want = [ref.surrogate_train_step(*p, update=stepped, lr=1e-6, want_grad=True) for _ in range(3)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    assert before > 8 * GB
    hog = torch.empty(before - 2 * GB, dtype=torch.uint8, device="cuda")
    try:
        left = torch.cuda.mem_get_info()[0]
        assert 1.7 * GB < left < 2.3 * GB
        got = [s.surrogate_train_step(*p, update=stepped, lr=1e-6, want_grad=True) for _ in range(3)]
        used = left - torch.cuda.mem_get_info()[0]
    finally:
        del hog
        torch.cuda.empty_cache()
    assert 1.0 * GB < used < 1.4 * GB     # one set
    for k, ((loss, g), (loss1, g1)) in enumerate(zip(got, want)):
        if stepped and k:   # Adam's first steps turn the order of sums in tiny entries into full steps
            assert abs(loss - loss1) <= 1e-3 * loss1
            continue
        assert abs(loss - loss1) <= 1e-10 * loss1
        assert np.linalg.norm(g - g1) <= 1e-5 * np.linalg.norm(g1)


def test_no_memory_at_all_is_reported_and_leaves_nothing_behind(env):  # noqa: F811
    torch, sph = env
    w = WL.drop_tank(2, (500, 510), drop_d_dx=120, seed=5, perturb=True)
    norm, flat = _norm(w), SL.init_weights(2, seed=6, out_scale=1.0)
    t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (w.x, w.u, w.rho)]
    p = [a.data_ptr() for a in t]
    s = sph.Simulation.from_workload(w)
    s.surrogate_init(flat, norm)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 3 * GB // 4, dtype=torch.uint8, device="cuda")
    try:
        left = torch.cuda.mem_get_info()[0]
        with pytest.raises(sph.SphError) as e:
            s.surrogate_train_step(*p, update=False)
        assert e.value.code == -2
        assert left - torch.cuda.mem_get_info()[0] < 0.1 * GB
    finally:
        del hog
        torch.cuda.empty_cache()
    loss, g = s.surrogate_train_step(*p, update=False, want_grad=True)
    assert np.isfinite(loss) and np.linalg.norm(g) > 0
