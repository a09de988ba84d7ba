"""The number of chunks that the row kernels' panels are split into: short rows of one warp
per CTA, of which more than eight fit an SM, few panels, odd counts, against the FP64
oracle; and launches that are full already, which are not split.

Tolerance: 1e-4 relative l2, the operators' bound everywhere."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


@pytest.mark.parametrize("nt,nx,nv,batch", [
    (100, 256, 9, 12), (50, 200, 12, 6), (20, 250, 12, 6),   # one warp per CTA: many fit an SM
    (200, 100, 16, 6), (200, 12, 3, 2), (40, 5, 2, 1), (100, 30, 32, 3),
    (400, 60, 3, 1), (400, 60, 16, 6), (1500, 8, 4, 3), (700, 20, 192, 2),
])
def test_split_of_short_and_many_rows(lib, nt, nx, nv, batch):
    from oracle import stolt
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1400.0, 3500.0, nv)
    plan = ashrt.Plan(nt, nx, DT, DX, v, max_batch=batch)
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)
    rng = np.random.default_rng(nt + nv)
    m = rng.standard_normal((batch,) + g.model_shape).astype(np.float32)
    d = rng.standard_normal((batch,) + g.data_shape).astype(np.float32)
    md, dd = torch.from_numpy(m).cuda(), torch.from_numpy(d).cuda()
    od, om = torch.full_like(dd, float("nan")), torch.full_like(md, float("nan"))
    plan.forward(md, od, batch=batch)
    plan.adjoint(dd, om, batch=batch)
    for b in (0, batch - 1):                        # 1e-4, the operators' bound everywhere
        rd, rm = stolt.forward(g, m[b].astype(np.float64)), stolt.adjoint(g, d[b].astype(np.float64))
        assert np.linalg.norm(od[b].cpu().numpy() - rd) <= 1e-4 * np.linalg.norm(rd)
        assert np.linalg.norm(om[b].cpu().numpy() - rm) <= 1e-4 * np.linalg.norm(rm)
    plan.close()


@pytest.mark.parametrize("nt,nx,nv,batch", [(100, 256, 9, 12), (20, 250, 12, 10), (50, 250, 10, 12)])
def test_full_launches_are_not_split(lib, nt, nx, nv, batch):
    """More than eight panels are added chunk by chunk, so the bits of a split forward are
    its own: those of these calls (six CTAs per SM and more, 26.7 us unsplit and 41.9 split
    for the first) are those of the same gathers in a call four times the size."""
    import torch
    from paper_1711_10214_gb300 import ashrt
    plan = ashrt.Plan(nt, nx, DT, DX, np.linspace(1400.0, 3500.0, nv), max_batch=4 * batch)
    gen = torch.Generator(device="cuda").manual_seed(2)
    m = torch.randn((4 * batch,) + plan.model_shape, device="cuda", generator=gen)
    few, many = (torch.empty((n,) + plan.data_shape, device="cuda") for n in (batch, 4 * batch))
    plan.forward(m, few, batch=batch)
    plan.forward(m, many, batch=4 * batch)
    assert torch.equal(few, many[:batch])
    plan.close()
