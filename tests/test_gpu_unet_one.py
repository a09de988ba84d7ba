"""Warm-start U-Net with one output channel (the weights' channel alone): the head writes
only its last channel, and the head's backward has a single channel in its block.

Tolerances: those of test_gpu_unet_train.py, 5e-3 for the loss and 1.5e-2 for a gradient,
were set with three and more channels.  What they allow for is activations that FP32
accumulation order moves across a BF16 boundary; a channel's share of loss and gradient
feels them independently of the others', so the relative error of a sum over C
channels falls with sqrt(C), and one channel has sqrt(3) times that of three: 9e-3 and
2.6e-2.  A prediction is the forward's output scaled, bit for bit."""
import numpy as np
import pytest

from oracle import unet

pytestmark = pytest.mark.gpu
Q = unet.bf16_round


def _flat(p, specs):
    return np.concatenate([np.concatenate([p[s[0] + ".w"].ravel(), p[s[0] + ".b"].ravel()])
                           for s in specs]).astype(np.float32)


def _unflat(v, specs):
    out, o = {}, 0
    for name, ci, co, k in specs:
        out[name + ".w"] = v[o:o + co * ci * k * k].reshape(co, ci, k, k).astype(np.float64)
        o += co * ci * k * k
        out[name + ".b"] = v[o:o + co].astype(np.float64)
        o += co
    return out


@pytest.mark.parametrize("H,W,n", [(32, 72, 2), (64, 64, 1), (16, 264, 2)])
def test_one_channel_training_step(lib, H, W, n):
    import torch
    from paper_1711_10214_gb300 import ashrt
    rng = np.random.default_rng(H * W + n)
    specs = unet.layer_specs(1, 1)
    p = unet.init_params(rng, 1, 1)
    for name, _, co, _ in specs:
        p[name + ".b"] = 0.05 * rng.standard_normal(co)
    flat = _flat(p, specs)
    p = _unflat(flat, specs)
    x = (3.0 * rng.standard_normal((n, H, W))).astype(np.float32)
    t = rng.standard_normal((n, 1, H, W)).astype(np.float32)
    lam = np.array([0.7], np.float32)
    net = ashrt.UNet(H, W, 1, max_batch=n, params=flat)
    loss = net.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), lr=0.0,
                          channel_weight=lam)
    got = _unflat(net.grads(), specs)
    net.close()
    x64 = x.astype(np.float64)
    xn = x64 / np.sqrt(np.mean(x64 * x64, axis=(1, 2)))[:, None, None]
    yq, cache = unet.forward(p, xn[:, None], 1, rnd=Q)
    lq, gy = unet.mse_loss(yq, t.astype(np.float64), lam)
    ref = unet.backward(p, cache, gy, rnd=Q, rnd_g=Q)
    assert abs(loss - lq) <= 9e-3 * lq
    for k in ref:
        assert np.linalg.norm(got[k] - ref[k]) <= 2.6e-2 * np.linalg.norm(ref[k]), k


@pytest.mark.parametrize("H,W,n,cout", [(32, 72, 2, 1), (8, 8, 1, 1), (16, 136, 3, 2), (8, 200, 2, 49)])
def test_prediction_is_the_forward_scaled(lib, H, W, n, cout):
    import torch
    from paper_1711_10214_gb300 import ashrt
    gen = torch.Generator(device="cuda").manual_seed(H + W)
    x = 2.0 * torch.randn((n, H, W), device="cuda", generator=gen)
    net = ashrt.UNet(H, W, cout, max_batch=n)
    y = torch.full((n, cout, H, W), float("nan"), device="cuda")
    net.forward(x, y, rescale=True, p=1.0)
    assert torch.isfinite(y).all()
    m0 = torch.full((n, max(cout - 1, 1), H, W), float("nan"), device="cuda")
    wr = torch.full((n, H, W), float("nan"), device="cuda")
    net.predict(x, m0 if cout > 1 else None, wr)
    assert torch.equal(wr, y[:, -1])
    if cout > 1:
        assert torch.equal(m0, y[:, :-1])
    # rescaled: the raw output times the RMS, and exp of the last channel over its root
    raw = torch.empty_like(y)
    net.forward(x, raw)
    rms = x.double().pow(2).mean(dim=(1, 2)).sqrt().float()[:, None, None]
    assert torch.allclose(wr, torch.exp(raw[:, -1]) / rms.sqrt(), rtol=1e-5, atol=0.0)
    net.close()
