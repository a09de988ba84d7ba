"""The time-domain pair on records of more than 2048 samples (512 threads per CTA) and
forwards of few panels, whose distances are dealt out over a cluster, against the FP64
oracle.

Tolerance: 1e-3 relative l2, as in test_gpu_timedomain_edges.py for more than 1024 samples
(the FP32 traveltime moves s by up to 5e-4 samples below 4096)."""
import numpy as np
import pytest

from oracle import timedomain

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5


@pytest.mark.parametrize("nt,nx,v,t0,batch", [
    (2049, 17, [2000.0], None, 1),                       # eight CTAs share the distances of a panel
    (4096, 9, [1500.0, 2500.0], None, 1),                # two panels, four each
    (4095, 2, [1800.0], None, 1),                        # two distances
    (3000, 40, [1500.0, 2000.0, 4000.0], [0.0, 0.4], 2), # six panels in four chunks
    (2500, 1, [1500.0, 2000.0], None, 3),                # one distance
    (2560, 100, list(np.linspace(1400.0, 3500.0, 9)), None, 1),   # 9 panels in eight chunks
    (1500, 20, [1700.0], None, 1), (2048, 5, [1700.0, 300.0, 2e5], None, 1),   # 256 threads
])
def test_long_records_match_oracle(lib, nt, nx, v, t0, batch):
    import torch
    from paper_1711_10214_gb300 import ashrt
    t0s = (0.0,) if t0 is None else t0
    rng = np.random.default_rng(nt + nx)
    m = rng.standard_normal((batch, len(t0s), len(v), nx, nt)).astype(np.float32)
    d = rng.standard_normal((batch, nx, nt)).astype(np.float32)
    md, dd = torch.from_numpy(m).cuda(), torch.from_numpy(d).cuda()
    od, om = torch.full_like(dd, np.nan), torch.full_like(md, np.nan)
    ashrt.td_forward(nt, nx, DT, DX, v, md, od, t0s=t0, batch=batch)
    ashrt.td_adjoint(nt, nx, DT, DX, v, dd, om, t0s=t0, batch=batch)
    again = torch.empty_like(od)
    ashrt.td_forward(nt, nx, DT, DX, v, md, again, t0s=t0, batch=batch)
    assert torch.equal(od, again)
    od, om = od.cpu().numpy().astype(np.float64), om.cpu().numpy().astype(np.float64)
    for b in range(batch):
        ref = timedomain.forward(nt, nx, DT, DX, v, m[b], t0s)
        assert np.linalg.norm(od[b] - ref) <= 1e-3 * np.linalg.norm(ref)
        ref = timedomain.adjoint(nt, nx, DT, DX, v, d[b], t0s).reshape(om[b].shape)
        assert np.linalg.norm(om[b] - ref) <= 1e-3 * np.linalg.norm(ref)
    lhs, rhs = np.vdot(od, d.astype(np.float64)), np.vdot(m.astype(np.float64), om)
    assert abs(lhs - rhs) <= 1e-5 * np.linalg.norm(od) * np.linalg.norm(d)


def _best_us(f, reps=20):
    import torch
    f()
    best = 1e9
    e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(reps):
        e0.record()
        f()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1))
    return best


def test_long_records_keep_the_rate(lib):
    """Time per (sample, panel, apex, trace) at 4096 samples within 1.6 times that at 2048:
    steps reach further on a longer record, so a little more of the work is left in it.
    With 16 samples per thread the ratio was over 2.5."""
    import torch
    from paper_1711_10214_gb300 import ashrt
    t = {}
    for nt in (2048, 4096):
        v = np.linspace(1400.0, 3500.0, 16)
        d = torch.randn((4, 128, nt), device="cuda")
        m = torch.empty((4, 1, 16, 128, nt), device="cuda")
        t[nt] = _best_us(lambda: ashrt.td_adjoint(nt, 128, DT, DX, v, d, m, batch=4), 5)
    assert t[4096] <= 2 * 1.6 * t[2048], t
