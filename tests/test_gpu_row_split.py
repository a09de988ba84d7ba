"""Row kernels whose panels are split over several CTAs (few rows) and the
choice of the row kernels' form by batch: the operator pair against the FP64
oracle, and the chosen form against a fixed one.

Tolerance: 1e-4 relative l2 against the oracle, the operators' bound
everywhere; two forms of the same operator differ by FP32 rounding of
transforms of length <= 4096 and sums of <= 72 panels, below 2e-6 (about 20
roundings of 6e-8 each)."""
import numpy as np
import pytest

from oracle import stolt

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nt,nx,nv,t0,batch", [
    (20, 5, 8, None, 1),                      # Nt 64: one panel per chunk
    (250, 12, 9, None, 3),                    # Nt 512: 9 panels in 8 chunks (2, 2, 2, 2, 1, 0, 0, 0)
    (256, 16, 3, [0.0, 0.02, 0.05], 2),       # chunks that begin inside a shift
    (130, 9, 1, None, 1),                     # one panel: no split
    (300, 10, 5, [0.0, 0.013], 1),            # Nt 1024, single-gather form
    (600, 12, 3, [0.0, 0.02, 0.05], 2),       # Nt 2048
    (1100, 6, 9, None, 1),                    # Nt 4096
    (1500, 5, 2, [0.0, 0.04, 0.1], 2),        # Nt 4096, shifts
])
def test_split_panels_match_oracle(lib, nt, nx, nv, t0, batch):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1500.0, 9000.0 if nv > 4 else 3000.0, nv)   # fast ones leave dead rows
    plan = ashrt.Plan(nt, nx, DT, DX, v, t0s=t0, max_batch=batch, wavelet_peak_hz=25.0)
    g = stolt.Geometry(nt, nx, DT, DX, v, t0s=(0.0,) if t0 is None else t0, Nt=plan.Nt, Nx=plan.Nx,
                       wavelet_peak_hz=25.0)
    rng = np.random.default_rng(nt + nx)
    m = rng.standard_normal((batch,) + g.model_shape).astype(np.float32)
    d = rng.standard_normal((batch,) + g.data_shape).astype(np.float32)
    md, dd = torch.from_numpy(m).cuda(), torch.from_numpy(d).cuda()
    od, om = torch.full_like(dd, float("nan")), torch.full_like(md, float("nan"))
    plan.forward(md, od, batch=batch)
    plan.adjoint(dd, om, batch=batch)
    torch.cuda.synchronize()
    assert _rel(od.cpu().numpy(), stolt.forward_batch(g, m)) <= 1e-4
    assert _rel(om.cpu().numpy(), stolt.adjoint_batch(g, d)) <= 1e-4
    plan.close()


@pytest.mark.parametrize("nt,nx,nv,nt0,batch,fixed", [
    (600, 60, 6, 1, 8, 9),       # Nt 2048, 520 rows
    (1000, 100, 6, 1, 7, 9),     # 903 rows: tensor-memory forward, single-gather adjoint
    (1000, 100, 4, 2, 16, 6),    # the same, shifts
    (1000, 250, 3, 1, 15, 9),    # 3855 rows: the pair form both ways
    (500, 40, 12, 6, 3, 4),      # Nt 1024, 72 panels
    (1500, 40, 6, 2, 5, 5),      # Nt 4096
])
def test_rule_matches_fixed_form(lib, nt, nx, nv, nt0, batch, fixed):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1400.0, 3500.0, nv)
    plan = ashrt.Plan(nt, nx, DT, DX, v, t0s=np.linspace(0.0, 0.2, nt0), max_batch=batch)
    gen = torch.Generator(device="cuda").manual_seed(5)
    m = torch.randn((batch,) + plan.model_shape, device="cuda", generator=gen)
    d = torch.randn((batch, nx, nt), device="cuda", generator=gen)
    out = []
    for variant in (None, fixed):
        if variant:
            plan.set_variant(variant, 16)
        od, om = torch.full_like(d, float("nan")), torch.full_like(m, float("nan"))
        plan.forward(m, od, batch=batch)
        plan.adjoint(d, om, batch=batch)
        torch.cuda.synchronize()
        out.append((od.double(), om.double()))
    for a, b in zip(out[0], out[1]):
        assert float((a - b).norm() / b.norm()) <= 2e-6
    plan.close()
