"""The irregular traces' contractions where their tiles (64 traces or 32
wavenumbers by 128 samples, chunks of eight) end, against the FP64 oracle.

Tolerance: 1e-4 relative l2 as for every operator test (FP32 sums of at most 257
products, below 2e-6)."""
import numpy as np
import pytest

from oracle import stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


@pytest.mark.parametrize("nt,nx,nr,batch,mask", [
    (127, 12, 63, 2, True),      # one short of a tile both ways, 17 wavenumbers
    (128, 16, 64, 1, False),     # whole tiles
    (129, 40, 65, 3, True),      # one more; 65 wavenumbers
    (33, 3, 1, 1, False),        # a single trace, fewer samples than a thread row
    (258, 100, 130, 2, False),   # 129 wavenumbers, three trace tiles
])
def test_irregular_tile_edges(lib, nt, nx, nr, batch, mask):
    import torch
    from paper_1711_10214_gb300 import ashrt
    rng = np.random.default_rng(nt + nr)
    x = rng.uniform(0.0, (nx - 1) * DX, nr)
    v = [1500.0, 2600.0]
    plan = ashrt.Plan(nt, nx, DT, DX, v, max_batch=batch, trace_x=x)
    g = stolt.Geometry(nt, nx, DT, DX, v, Nt=plan.Nt, Nx=plan.Nx)   # (Nx is 16 at least)
    m = rng.standard_normal((batch,) + g.model_shape).astype(np.float32)
    d = rng.standard_normal((batch, nr, nt)).astype(np.float32)
    mk = (rng.random((batch, nr)) < 0.7).astype(np.float32) if mask else None
    md, dd = torch.from_numpy(m).cuda(), torch.from_numpy(d).cuda()
    mkd = None if mk is None else torch.from_numpy(mk).cuda()
    od, om = torch.full_like(dd, float("nan")), torch.full_like(md, float("nan"))
    plan.forward(md, od, mask=mkd, batch=batch)
    plan.adjoint(dd, om, mask=mkd, batch=batch)
    rel = lambda a, b: float(np.linalg.norm(a - b) / np.linalg.norm(b))
    for b in range(batch):
        mb = None if mk is None else mk[b].astype(np.float64)
        assert rel(od[b].cpu().numpy(), stolt.forward_irregular(g, m[b].astype(np.float64), x, mb)) <= 1e-4
        assert rel(om[b].cpu().numpy(), stolt.adjoint_irregular(g, d[b].astype(np.float64), x, mb)) <= 1e-4
    plan.close()
