"""The row kernels' form by rule on both sides of its lines: which form ran
is read from the result's bits (a fixed variant gives the same ones), and the result is
compared with the other form's.  The 32 x 32 forward of 9 has its own bits, 6 and 8 share
theirs; the adjoints of 6 and 9 differ with asymptote shifts only.

Tolerance: two forms differ by FP32 rounding of transforms of length 2048 and sums of at
most 48 panels, 2e-6 (see test_gpu_row_split.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


def _pair(plan, batch, variant=None):
    import torch
    if variant:
        plan.set_variant(variant, 16)
    gen = torch.Generator(device="cuda").manual_seed(17)
    m = torch.randn((batch,) + plan.model_shape, device="cuda", generator=gen)
    d = torch.randn((batch,) + plan.data_shape, device="cuda", generator=gen)
    od, om = torch.full_like(d, float("nan")), torch.full_like(m, float("nan"))
    plan.forward(m, od, batch=batch)
    plan.adjoint(d, om, batch=batch)
    return od, om


@pytest.mark.parametrize("nx,nv,nt0,batch,fwd,adj", [
    (100, 1, 1, 4, 6, 6), (250, 1, 1, 16, 8, 8),       # one panel (257 rows: 4112)
    (100, 4, 1, 4, 6, 6), (100, 5, 1, 4, 9, 6),        # 129 rows: R P 2064, 2580
    (100, 7, 1, 3, 6, 6), (100, 9, 1, 3, 9, 6),        # an odd batch counts three quarters
    (16, 32, 1, 4, 6, 6), (16, 36, 1, 4, 9, 6),        # 17 rows: 2176, 2448
    (250, 8, 1, 16, 9, 6), (250, 9, 1, 16, 9, 9),      # 4112 rows: more than 8 panels
    (250, 9, 1, 14, 9, 6),                             # 3598 rows
    (250, 4, 3, 2, 9, 9), (250, 4, 3, 3, 9, 6),        # shifts: 257 pairs; three gathers
    (100, 8, 3, 6, 9, 9), (100, 8, 3, 8, 9, 6), (100, 8, 3, 10, 9, 9),   # 387, 516, 645 pairs
    (60, 8, 3, 6, 9, 6),                               # 195 pairs
])
def test_form_by_rule(lib, nx, nv, nt0, batch, fwd, adj):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.linspace(1400.0, 3500.0, nv) if nv > 1 else [2000.0]
    plan = ashrt.Plan(700, nx, DT, DX, v, t0s=np.linspace(0.0, 0.2, nt0) if nt0 > 1 else None,
                      max_batch=batch)
    assert plan.Nt == 2048
    od, om = _pair(plan, batch)
    for variant in (fwd, 6 if fwd == 9 else 9):
        fd, fm = _pair(plan, batch, variant)
        assert torch.equal(od, fd) == ((variant == 9) == (fwd == 9)), variant
        assert torch.equal(om, fm) == (nt0 == 1 or (variant == 9) == (adj == 9)), variant
        assert float((od - fd).norm() / fd.norm()) <= 2e-6
        assert float((om - fm).norm() / fm.norm()) <= 2e-6
    plan.close()
