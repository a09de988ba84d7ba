"""The path s = tau0 / dt + sqrt(tau^2 + h^2) of the time-domain pair, read back to the
last bit: with two traces, zeros on the first and d[t] = t mod 2 on the second, the
adjoint at the first apex is the weight that the sample floor(s) or floor(s) + 1 gets at
distance 1, which is f = s - floor(s) or 1 - f, both exact in FP32.  The square root has
to be the correctly rounded one, equal to CUDA's sqrtf (through torch) bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
f32 = np.float32


def _check(nt, dx, dt, v, t0=None):
    import torch
    from paper_1711_10214_gb300 import ashrt
    v = np.asarray(v, f32)
    t0s = np.asarray([0.0] if t0 is None else t0, f32)
    d = torch.zeros((1, 2, nt), device="cuda")
    d[0, 1] = torch.arange(nt, device="cuda") % 2
    m = torch.full((1, t0s.size, v.size, 2, nt), float("nan"), device="cuda")
    ashrt.td_adjoint(nt, 2, dt, dx, v, d, m, t0s=None if t0 is None else t0s)
    got = m[0, :, :, 0].cpu().numpy()
    cv = (dx / (v.astype(np.float64) * dt)).astype(f32)
    hs2 = cv * cv
    tau = np.arange(nt, dtype=np.float64)
    x64 = tau * tau + hs2.astype(np.float64)[:, None]
    x = x64.astype(f32)
    # (in FP64 the sum is exact to 53 bits: leave out what that rounding could tip over
    # the middle of two floats, and the roots that count as zero)
    up, down = np.nextafter(x, f32(np.inf)), np.nextafter(x, f32(0))
    ok = np.ones(x.shape, bool)
    for nb in (up, down):
        mid = 0.5 * (x.astype(np.float64) + nb.astype(np.float64))
        ok &= np.abs(x64 - mid) > 1e-15 * x64
    ok &= x > 1e-30
    q = torch.sqrt(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(q, np.sqrt(x))
    n = 0
    for j, t in enumerate(t0s):
        s = f32(np.float64(t) / dt) + q
        i0 = np.floor(s)
        f = (s - i0).astype(f32)
        odd = np.mod(i0, 2) == 1
        want = np.where(odd, f32(1) - f, f).astype(f32)
        want[(i0 >= nt) | (~odd & (i0 + 1 >= nt))] = 0.0
        bad = ok & (got[j] != want)
        assert not bad.any(), (t, x[bad][:5], q[bad][:5], got[j][bad][:5], want[bad][:5])
        n += int((ok & (i0 < nt)).sum())
    assert n > 0


def test_perfect_squares_and_their_neighbours(lib):
    # h = 5040 / v: whole numbers (tau^2 + h^2 has its Pythagorean squares), and the
    # velocities next to them
    v = np.array([k for k in range(2, 5041) if 5040 % k == 0], f32)
    v = np.concatenate([v, np.nextafter(v, f32(0)), np.nextafter(v, f32(np.inf))])
    _check(4096, 5040.0, 1.0, v)


@pytest.mark.parametrize("seed,nt", [(0, 4096), (1, 4096), (2, 4096), (3, 2048), (4, 1000), (5, 257)])
def test_every_binade(lib, seed, nt):
    rng = np.random.default_rng(seed)
    _check(nt, 1.0, 1.0, 2.0 ** rng.uniform(-12.0, 30.0, 256))


def test_fine_steps(lib):
    # h^2 in steps of a few ulp: consecutive floats x at tau = 1 and 2
    one = np.nextafter(f32(1), f32(2)) - f32(1)
    for base in (1.0, 1.2, 1.7, 2.0, 3.3):
        _check(64, 1.0, 1.0, f32(base) * (1 + np.arange(256, dtype=f32) * one))


def test_with_shifts(lib):
    v = 2.0 ** np.random.default_rng(9).uniform(-11.0, 4.0, 32)
    _check(3000, 1.0, 1.0, v, t0=[0.0, 0.37, 5.125, 100.3, 1999.99, 2999.5])
