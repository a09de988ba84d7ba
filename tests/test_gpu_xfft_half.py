"""Trace-axis analysis of panels that fill at most half of the padded axis
(Nx 256, 512 and 1024): the operator pair at the edges of each length (one trace
above the shorter length, exactly half, odd and even sample counts, a ragged
last column tile), the unpadded axis beside it (the general kernel), and the
fused CGLS updates of rows that the TMA kernel does not take, against the FP64
oracle.

Tolerances: 1e-4 relative l2 for the operators and 1e-3 for the recovered
gather, as everywhere."""
import numpy as np
import pytest

from oracle import irls, stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nt,nx,pad_x,Nx", [
    (33, 65, 2, 256), (40, 128, 2, 256), (33, 129, 2, 512), (34, 256, 2, 512),
    (33, 257, 2, 1024), (31, 512, 2, 1024),
    (33, 200, 1, 256), (34, 512, 1, 512), (33, 513, 1, 1024),      # more than half: general kernel
])
def test_operator_pair_matches_oracle(lib, nt, nx, pad_x, Nx):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v, B = [1500.0, 2600.0], 2
    plan = ashrt.Plan(nt, nx, DT, DX, v, max_batch=B, pad_x=pad_x)
    assert plan.Nx == Nx
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)
    rng = np.random.default_rng(nt * nx)
    m = rng.standard_normal((B,) + g.model_shape).astype(np.float32)
    d = rng.standard_normal((B,) + g.data_shape).astype(np.float32)
    mk = (rng.random((B, nx)) < 0.6).astype(np.float32)
    md, dd, mkd = (torch.from_numpy(x).cuda() for x in (m, d, mk))
    for cols in (16, 8):
        plan.set_variant(3, cols)
        od, om = torch.full_like(dd, float("nan")), torch.full_like(md, float("nan"))
        plan.forward(md, od, mask=mkd, batch=B)
        plan.adjoint(dd, om, mask=mkd, batch=B)
        torch.cuda.synchronize()
        assert _rel(od.cpu().numpy(), stolt.forward_batch(g, m, mk)) <= 1e-4
        assert _rel(om.cpu().numpy(), stolt.adjoint_batch(g, d, mk)) <= 1e-4
    plan.close()


@pytest.mark.parametrize("nt,nx", [(33, 70), (34, 130), (36, 300)])
def test_fused_updates_match_oracle(lib, nt, nx):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = [1500.0, 2600.0]
    plan = ashrt.Plan(nt, nx, DT, DX, v, with_solver=True)
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)
    rng = np.random.default_rng(nx)
    d = stolt.forward(g, rng.standard_normal(g.model_shape))
    d = (d + 5.0 * d.std() * (rng.random(d.shape) < 0.02)).astype(np.float32)
    dd = torch.from_numpy(d[None]).cuda()
    m = torch.empty((1,) + plan.model_shape, device="cuda")
    drec = torch.empty_like(dd)
    plan.deblend(dd, m, drec=drec, n_outer=2, n_cg=5)
    mo, rep = irls.irls(lambda x: stolt.forward(g, x), lambda x: stolt.adjoint(g, x), d, 2, 5)
    assert _rel(drec[0].cpu().numpy(), rep["d_model"]) <= 1e-3
    assert _rel(m[0].cpu().numpy(), mo) <= 1e-3
    plan.close()
