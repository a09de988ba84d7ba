"""Forward rows at Nt 2048 in the 32 x 32 form (tensor-memory forward, nt <= Nt / 2)
and beside its limits: the operator against the FP64 oracle.

Tolerance: 1e-4 relative l2 as for every operator test; the transforms, the map and
the sum over the panels are FP32 (about 30 roundings of 6e-8 each, below 2e-6)."""
import numpy as np
import pytest

from oracle import stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


@pytest.mark.parametrize("nt,nx,nv,t0,batch,pad_t", [
    (1024, 5, 3, None, 2, 2),                 # every row full
    (1023, 9, 2, None, 3, 2),                 # a group of rows short by one, an odd batch
    (513, 4, 1, None, 1, 2),                  # the shortest rows, one panel, no second gather
    (769, 12, 3, [0.0, 0.02, 0.05], 5, 2),    # a group's first sample only, shifts
    (600, 16, 3, [0.0, 0.02, 0.05], 2, 2),    # 9 panels in 8 chunks that begin inside a shift
    (1025, 6, 2, None, 2, 1),                 # longer than Nt / 2: the 16 x 16 x 8 form
    (2048, 5, 2, [0.0, 0.03], 3, 1),
])
def test_forward_2048_matches_oracle(lib, nt, nx, nv, t0, batch, pad_t):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1500.0, 9000.0, nv) if nv > 1 else np.array([2000.0])
    plan = ashrt.Plan(nt, nx, DT, DX, v, t0s=t0, max_batch=batch, pad_t=pad_t)
    assert plan.Nt == 2048
    plan.set_variant(9, 16)
    g = stolt.Geometry(nt, nx, DT, DX, v, t0s=(0.0,) if t0 is None else t0, Nt=plan.Nt, Nx=plan.Nx)
    m = np.random.default_rng(nt).standard_normal((batch,) + g.model_shape).astype(np.float32)
    md = torch.from_numpy(m).cuda()
    od = torch.full((batch,) + g.data_shape, float("nan"), device="cuda")
    plan.forward(md, od, batch=batch)
    ref = stolt.forward_batch(g, m)
    got = od.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    plan.close()
