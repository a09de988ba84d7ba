"""The irregular traces' contractions in their three tile sizes.  A sum runs over its
wavenumbers or traces in ascending order whatever the tile, so the same gather gives
the same bits alone (small tiles), among a few and in a launch that fills the chip with
the largest ones; alone it is compared with the FP64 oracle as well.

Tolerance: 1e-4 relative l2, the operators' bound everywhere."""
import numpy as np
import pytest

from oracle import stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


@pytest.mark.parametrize("nt,nx,nr", [
    (31, 6, 5), (33, 6, 33), (64, 16, 32), (65, 20, 31), (129, 30, 65), (191, 40, 64),
    (192, 70, 130), (200, 130, 129), (255, 16, 1),
])
@pytest.mark.parametrize("mask", [False, True])
def test_tiles_agree(lib, nt, nx, nr, mask):
    import torch
    from paper_1711_10214_gb300 import ashrt
    rng = np.random.default_rng(nt + nr)
    x = np.sort(rng.uniform(0.0, (nx - 1) * DX, nr))
    B = 400
    plan = ashrt.Plan(nt, nx, DT, DX, [2100.0], max_batch=B, trace_x=x)
    gen = torch.Generator(device="cuda").manual_seed(nr)
    m = torch.randn((B,) + plan.model_shape, device="cuda", generator=gen)
    d = torch.randn((B, nr, nt), device="cuda", generator=gen)
    mk = (torch.rand((B, nr), device="cuda", generator=gen) < 0.7).float() if mask else None
    out = {}
    for n in (1, 2, 7, 30, 90, B):
        od, om = torch.full_like(d[:n], float("nan")), torch.full_like(m[:n], float("nan"))
        plan.forward(m, od, mask=mk, batch=n)
        plan.adjoint(d, om, mask=mk, batch=n)
        out[n] = od, om
    for n in (2, 7, 30, 90, B):
        assert torch.equal(out[n][0][:1], out[1][0]) and torch.equal(out[n][1][:1], out[1][1]), n
    g = stolt.Geometry(nt, nx, DT, DX, [2100.0], Nt=plan.Nt, Nx=plan.Nx)
    mb = None if mk is None else mk[0].cpu().numpy().astype(np.float64)
    rd = stolt.forward_irregular(g, m[0].cpu().numpy().astype(np.float64), x, mb)
    rm = stolt.adjoint_irregular(g, d[0].cpu().numpy().astype(np.float64), x, mb)
    assert np.linalg.norm(out[1][0][0].cpu().numpy() - rd) <= 1e-4 * np.linalg.norm(rd)
    assert np.linalg.norm(out[1][1][0].cpu().numpy() - rm) <= 1e-4 * np.linalg.norm(rm)
    plan.close()
