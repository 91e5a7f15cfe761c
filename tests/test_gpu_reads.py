"""One field read into pinned host memory (written in place, vectors in whole
lines) gives the bits of the staged read into a pageable array: at a count whose
last 256-particle tile is ragged and holds an odd number of doubles, at starts 8
and 4 bytes off a 16-byte boundary (staged), and for fields that stay staged.
"""
import numpy as np
import pytest

from paper_1702_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

FIELDS = ["pos", "vel", "acc", "rho", "rho_eval", "pressure", "drho", "tensor", "cell"]


@pytest.mark.parametrize("offset", [0, 8, 4])
@pytest.mark.parametrize("dim", [2, 3])
def test_pinned_field_reads_match_staged_reads(dim, offset):
    import torch
    from paper_1702_07760_gb300 import sph
    w = (WL.drop_tank(2, (37, 53), drop_d_dx=10, seed=21, perturb=True) if dim == 2
         else WL.drop_tank(3, (13, 17, 19), drop_d_dx=8, seed=22, perturb=True))
    assert w.n % 2 == 1 and w.n % 256 != 0
    sim = sph.Simulation.from_workload(w)
    sim.run(WL.stable_dt(w.params), 3)
    sim.eval_rates()
    for f in FIELDS:
        want = sim.read(f)
        raw = torch.zeros(want.nbytes + 64, dtype=torch.uint8, pin_memory=True).numpy()
        out = np.ndarray(want.shape, want.dtype, buffer=raw, offset=offset)
        assert out.ctypes.data % 16 == offset
        sim.read(f, out=out)
        assert np.array_equal(out, want), f
        assert not raw[:offset].any() and not raw[offset + want.nbytes:].any(), f
    sim.close()
