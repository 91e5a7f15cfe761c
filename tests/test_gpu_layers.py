"""The layer contraction (K whole in shared memory) at the edges of its tiles
and against the general one, and the weight gradients at the edges of their
chunks of 64 and splits of 4 096 nodes.

The layer path takes outputs on 16-byte boundaries; the same product into rows
of an odd length goes through the general path.  Both accumulate K in the same
order, so they agree bit for bit; against an FP32 product the bound is a few
FP32 ulps of K terms of |a b| (as for the general path).
"""
import numpy as np
import pytest

from oracle import mpnn as O
from paper_1702_07760_gb300 import surrogate_layout as SL
from paper_1702_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1702_07760_gb300 import build as B
    from paper_1702_07760_gb300 import sph
    B.build()
    sph.load()
    torch.cuda.set_device(0)
    return torch, sph


@pytest.mark.parametrize("N,K", [(128, 16), (128, 128), (128, 256), (256, 128), (16, 128)])
# one row, around one tile, and more tiles than two blocks an SM (304) take at once
@pytest.mark.parametrize("M", [1, 127, 128, 129, 128 * 304 + 5])
def test_layer_matches_the_general_contraction(env, M, N, K):
    torch, sph = env
    g = torch.Generator().manual_seed(M + N + K)
    A = (torch.randn(M, K, generator=g) * 0.5).to(torch.bfloat16)
    B = (torch.randn(N, K, generator=g) * 0.5).to(torch.bfloat16)
    dA, dB = A.cuda(), B.cuda()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    out = []
    for ldc in (N, N + 1):
        C = torch.full((M, ldc), -7.0, device="cuda")
        sph.mm_bf16(dA.data_ptr(), K, dB.data_ptr(), K, C.data_ptr(), ldc, M, N, K, 0, False, s, err.data_ptr())
        torch.cuda.synchronize()
        out.append(C[:, :N].cpu())
        assert torch.all(C[:, N:] == -7.0)
    assert int(err.item()) == 0
    assert torch.equal(out[0], out[1])
    ref = A.float() @ B.float().T
    bound = (A.float().abs() @ B.float().abs().T) * (K * 2.0 ** -22) + 1e-30
    assert torch.all((out[0] - ref).abs() <= bound)


# 143 nodes = 2 chunks and 15, 4 095 = a split less a node, 4 225 = a split and 2 chunks and a node, and 3-D
@pytest.mark.parametrize("shape", [(5, 7), (59, 57), (59, 59), (4, 5, 7)])
def test_gradient_sizes(env, shape):
    """As test_gradients_match_oracle (BF16 operands: cosine above 0.999 and relative
    norm error below 2e-2 over the whole gradient), at sizes around the chunk edges."""
    torch, sph = env
    dim = len(shape)
    w = WL.drop_tank(dim, shape, drop_d_dx=3, seed=sum(shape), perturb=True, quantise=16)
    rng = np.random.Generator(np.random.PCG64(sum(shape)))
    c0 = w.params["c0"]
    mu_in = np.concatenate([np.zeros(dim), [1e-4], [0, 0], np.zeros(dim), [0]])
    sd_in = np.concatenate([np.full(dim, 0.006 * c0), [1e-3], [1, 1], np.full(dim, 0.05), [1e-3]])
    sd_out = np.concatenate([np.full(dim, 1e-6), np.full(dim, 1e-2), [1e-4]])
    k_ref = 20.0 if dim == 2 else 80.0
    norm = SL.make_norm(dim, mu_in, sd_in, np.zeros(2 * dim + 1), sd_out, k_ref, 8 * WL.stable_dt(w.params),
                        0.008 * c0, 1.5e-3)
    flat = SL.init_weights(dim, seed=3, out_scale=1.0)
    rho0 = np.asarray(w.params["rho0"])[w.phase]
    fl = (w.wall == 0)[:, None]
    x1 = w.x + fl * rng.normal(0, 1, w.x.shape) * sd_out[:dim]
    u1 = w.u + fl * rng.normal(0, 1, w.u.shape) * sd_out[dim:2 * dim]
    r1 = w.rho + rng.normal(0, 1, w.n) * sd_out[2 * dim] * rho0
    t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x1, u1, r1)]
    sim = sph.Simulation.from_workload(w)
    sim.surrogate_init(flat, norm)
    grads = [sim.surrogate_train_step(*[a.data_ptr() for a in t], update=False, want_grad=True)[1] for _ in range(2)]
    recv, send, E = O.graph(w.params, w.x, w.phase, w.u, w.rho, norm)
    a, drdt = O.rates(w.params, w.x, w.u, w.rho, w.phase, w.wall)
    X = O.node_features(w.params, w.u, w.rho, w.phase, w.wall, norm, a, drdt)
    y, cache = O.forward(flat, dim, X, E, recv, send, k_ref)
    tt = O.targets(w.params, w.x, w.u, w.rho, x1, u1, r1, w.phase, norm, a, drdt)
    _, dy = O.loss(y, tt, O.output_mask(dim, w.wall))
    gr = O.backward(flat, dim, cache, dy)
    for g in grads:
        assert g @ gr / (np.linalg.norm(g) * np.linalg.norm(gr)) > 0.999
        assert np.linalg.norm(g - gr) / np.linalg.norm(gr) < 2e-2
    # the same state again: only the order of the FP32 atomics differs
    assert np.linalg.norm(grads[1] - grads[0]) < 1e-5 * np.linalg.norm(gr)


@pytest.mark.parametrize("dim", [2, 3])
def test_weight_gradients_of_partly_filled_rows(env, dim):
    """The decoder's gradient has 5 or 7 rows, so most lanes of the warps that store it have
    none: each tensor with its own error, within the 3e-2 that BF16 operands leave an output."""
    from test_gpu_surrogate import _case
    torch, sph = env
    w, norm, flat = _case(dim, 60 + dim)
    rng = np.random.Generator(np.random.PCG64(61))
    _, _, _, sd_out = SL.split_norm(norm, dim)[:4]
    fl = (w.wall == 0)[:, None]
    x1 = w.x + fl * rng.normal(0, 1, w.x.shape) * sd_out[:dim]
    u1 = w.u + fl * rng.normal(0, 1, w.u.shape) * sd_out[dim:2 * dim]
    r1 = w.rho + rng.normal(0, 1, w.n) * sd_out[2 * dim] * np.asarray(w.params["rho0"])[w.phase]
    t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x1, u1, r1)]
    sim = sph.Simulation.from_workload(w)
    sim.surrogate_init(flat, norm)
    _, g = sim.surrogate_train_step(*[a.data_ptr() for a in t], update=False, want_grad=True)
    recv, send, E = O.graph(w.params, w.x, w.phase, w.u, w.rho, norm)
    a, drdt = O.rates(w.params, w.x, w.u, w.rho, w.phase, w.wall)
    X = O.node_features(w.params, w.u, w.rho, w.phase, w.wall, norm, a, drdt)
    y, cache = O.forward(flat, dim, X, E, recv, send, 20.0 if dim == 2 else 80.0)
    tt = O.targets(w.params, w.x, w.u, w.rho, x1, u1, r1, w.phase, norm, a, drdt)
    _, dy = O.loss(y, tt, O.output_mask(dim, w.wall))
    want = SL.unflatten(O.backward(flat, dim, cache, dy), dim)
    got = SL.unflatten(g, dim)
    for name in ("dec2.w", "enc1.w"):
        assert np.linalg.norm(got[name] - want[name]) < 3e-2 * np.linalg.norm(want[name]), name


@pytest.mark.parametrize("M", [5, 31, 33, 100])
@pytest.mark.parametrize("N", [64, 128, 256])
def test_ragged_rows_over_several_column_chunks(env, M, N):
    """The general contraction with a last tile of few rows and several chunks of 16 columns a
    warp; rows of an odd length and K = 48 keep it off the layer path."""
    torch, sph = env
    K = 48
    g = torch.Generator().manual_seed(M * N)
    A = (torch.randn(M, K, generator=g) * 0.5).to(torch.bfloat16)
    B = (torch.randn(N, K, generator=g) * 0.5).to(torch.bfloat16)
    dA, dB = A.cuda(), B.cuda()
    C = torch.full((M + 1, N + 1), -7.0, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    sph.mm_bf16(dA.data_ptr(), K, dB.data_ptr(), K, C.data_ptr(), N + 1, M, N, K, 0, False,
                torch.cuda.current_stream().cuda_stream, err.data_ptr())
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert torch.all(C[M] == -7.0) and torch.all(C[:, N] == -7.0)
    ref = A.float() @ B.float().T
    bound = (A.float().abs() @ B.float().abs().T) * (K * 2.0 ** -22) + 1e-30
    assert torch.all((C[:M, :N].cpu() - ref).abs() <= bound)
