"""Warm-start U-Net on gathers of any amplitude: the RMS that normalises a gather and
the training loss are sums of squares that leave FP32's range long before the values
do, so both are formed in FP64.  Scaling a gather by a power of two scales its RMS by
exactly that power and changes nothing else.

Tolerances: the normalised outputs of the scaled gather are those of the gather itself
but for the last bit of an FP32 RMS (the FP64 partial sums meet in any order), which can
move a few BF16 roundings of the image: 2^-9, the BF16 unit roundoff.  The loss against an
FP64 sum of the same outputs: a thread adds n = pixels * images * channels /
(threads) terms, below 1e4 roundings of 2^-53 each, 1e-12."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H, W, COUT, N = 16, 40, 5, 2


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("log2", [-90, -83, -73, -64, 0, 61, 66, 100])
def test_gather_scale(lib, log2):
    import torch
    from paper_1711_10214_gb300 import ashrt
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((N, H, W), device="cuda", generator=gen)
    s = 2.0 ** log2
    net = ashrt.UNet(H, W, COUT, max_batch=N)
    y, ys = (torch.empty((N, COUT, H, W), device="cuda") for _ in range(2))
    net.forward(x, y)
    net.forward(x * s, ys)
    assert _rel(ys, y) <= 2.0 ** -9
    # in input units: the panels scale with the gather, the weights (p = 1) with s^(-1/2)
    m, ms = (torch.empty((N, COUT - 1, H, W), device="cuda") for _ in range(2))
    w, ws = (torch.empty((N, H, W), device="cuda") for _ in range(2))
    net.predict(x, m, w)
    net.predict(x * s, ms, ws)
    assert _rel(ms.double() / s, m) <= 2.0 ** -9
    assert _rel(ws.double() * s ** 0.5, w) <= 2.0 ** -9
    # targets: panels over the RMS, log of the weights in normalised units
    t, ts = (torch.empty((N, COUT, H, W), device="cuda") for _ in range(2))
    net.targets(x, m, w, t)
    net.targets(x * s, ms, ws, ts)
    assert _rel(ts, t) <= 2.0 ** -9
    # a training step sees the same image
    tg = torch.randn((N, COUT, H, W), device="cuda", generator=gen)
    loss = net.train_step(x, tg, lr=0.0)
    grads = net.grads()
    assert abs(net.train_step(x * s, tg, lr=0.0) - loss) <= 2.0 ** -9 * loss
    g = net.grads()
    assert np.linalg.norm(g - grads) <= 2.0 ** -6 * np.linalg.norm(grads)
    net.close()


@pytest.mark.parametrize("scale,weight", [(1.0, 1.0), (1.0, 0.3), (1e20, 1.0), (1e25, 1e-3), (1.0, 1e-30)])
def test_loss_is_an_fp64_sum(lib, scale, weight):
    import torch
    from paper_1711_10214_gb300 import ashrt
    gen = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn((N, H, W), device="cuda", generator=gen)
    t = torch.randn((N, COUT, H, W), device="cuda", generator=gen) * scale
    lam = (weight * np.linspace(0.5, 1.5, COUT)).astype(np.float32)
    net = ashrt.UNet(H, W, COUT, max_batch=N)
    y = torch.empty_like(t)
    net.forward(x, y)
    e = (y - t).double()
    want = float(((e * e).mean(dim=(0, 2, 3)) * torch.from_numpy(lam).cuda().double()).sum())
    loss = net.train_step(x, t, lr=0.0, channel_weight=lam)
    assert abs(loss - want) <= 1e-12 * want
    net.close()
