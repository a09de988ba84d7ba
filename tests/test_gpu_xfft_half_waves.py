"""The half-length trace-axis analysis with the fused CGLS update, which is taken from
six waves of CTAs on, and the launches just below that: robust deblending of many tiny
gathers at Nx 256, 512 and 1024, the first and the last against the FP64 oracle's
IRLS.

Tolerance: 1e-3 relative l2, the deblend's bound everywhere."""
import numpy as np
import pytest

from oracle import irls, stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nt,nx,pad_x,Nx,batch", [
    (35, 6, 40, 256, 228),       # 3648 tiles of 32 columns: the first launch that takes it
    (34, 6, 64, 512, 114),       # 1824 tiles
    (34, 6, 64, 512, 113),       # 1808: the length-N kernel
    (33, 6, 128, 1024, 76),      # 1824 tiles of 16 columns, a ragged one
])
def test_fused_updates_of_many_gathers(lib, nt, nx, pad_x, Nx, batch):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1500.0, 2900.0, 8)
    plan = ashrt.Plan(nt, nx, DT, DX, v, pad_x=pad_x, max_batch=batch, with_solver=True)
    assert plan.Nx == Nx
    plan.set_variant(3, 16)
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)
    rng = np.random.default_rng(Nx + batch)
    d = rng.standard_normal((batch, nx, nt)).astype(np.float32)
    dd = torch.from_numpy(d).cuda()
    m = torch.empty((batch,) + plan.model_shape, device="cuda")
    drec = torch.empty_like(dd)
    plan.deblend(dd, m, drec=drec, batch=batch, n_outer=2, n_cg=5)
    for b in (0, batch - 1):
        mo, rep = irls.irls(lambda x: stolt.forward(g, x), lambda x: stolt.adjoint(g, x),
                            d[b].astype(np.float64), 2, 5)
        assert _rel(drec[b].cpu().numpy(), rep["d_model"]) <= 1e-3
        assert _rel(m[b].cpu().numpy(), mo) <= 1e-3
    plan.close()
