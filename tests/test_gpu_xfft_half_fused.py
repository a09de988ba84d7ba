"""The half-length trace-axis analysis with the fused CGLS updates on gathers that fill
half of the padded axis, in launches of six waves of CTAs (fewer take the length-N
kernel): every row group of the update and both butterflies of N 1024 see data, and the
data-side update as well as the model-side one, since with one panel both launches have
the same tiles.  nx half the axis, one less, and one more than a quarter; even and odd
nt (rows that the TMA kernel does not take); both column tiles.  The first, a middle and
the last gather against the FP64 oracle's IRLS.

Tolerance: 1e-3 relative l2, the deblend's bound everywhere."""
import numpy as np
import pytest

from oracle import irls, stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("cols", [16, 8])
@pytest.mark.parametrize("nt,nx,Nx", [
    (130, 128, 256), (131, 127, 256), (129, 65, 256),
    (130, 256, 512), (129, 255, 512), (131, 129, 512),
    (132, 512, 1024), (129, 511, 1024), (130, 257, 1024),
])
def test_fused_updates_on_full_gathers(lib, nt, nx, Nx, cols):
    import torch
    from paper_1711_10214_gb300 import ashrt
    c = cols if Nx < 1024 else 8
    waves = 6 * 152 * (512 // (Nx * c // 32))
    per = (nt + 2 * c - 1) // (2 * c)
    batch = (waves + per - 1) // per + 3
    v = [2100.0]
    plan = ashrt.Plan(nt, nx, DT, DX, v, max_batch=batch, with_solver=True)
    assert plan.Nx == Nx and plan.P == 1
    plan.set_variant(3, cols)
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)
    gen = torch.Generator(device="cuda").manual_seed(Nx + nt)
    d = torch.randn((batch, nx, nt), device="cuda", generator=gen)
    m = torch.empty((batch,) + plan.model_shape, device="cuda")
    drec = torch.empty_like(d)
    plan.deblend(d, m, drec=drec, batch=batch, n_outer=2, n_cg=5)
    for b in (0, batch // 2, batch - 1):
        mo, rep = irls.irls(lambda x: stolt.forward(g, x), lambda x: stolt.adjoint(g, x),
                            d[b].cpu().numpy().astype(np.float64), 2, 5)
        assert _rel(drec[b].cpu().numpy(), rep["d_model"]) <= 1e-3
        assert _rel(m[b].cpu().numpy(), mo) <= 1e-3
    plan.close()
