"""Workloads of the library as a user's program runs them, for timing.

A case is a dict of plain values with a "kind", which names the entry points it
goes through:

  pair     Plan.forward and Plan.adjoint, the operator pair (regular or
           irregular traces, with or without asymptote shifts, wavelet, band
           limit and trace mask)
  deblend  Plan.deblend, the robust IRLS / CGLS solve
  batch    Batch.deblend, the solve of gathers of uneven trace counts
  fista    Plan.fista, the sparse inversion of decimated AASHRT gathers
  td       td_forward and td_adjoint, the time-domain (hyperbolic) pair
  predict  UNet.predict, the learned warm start at inference
  train    UNet.train_step, one training step of the warm start
  cube     blend, pseudo_deblend and sort_gathers, the acquisition model

prepare() makes what the program has before the call (inputs on the GPU, the
plan or the network), run() is the call, exact() the same numbers in FP64 by
plain torch.
"""
import math

import numpy as np
import torch

from paper_1711_10214_gb300 import ashrt

DT, DX = 0.004, 12.5          # 4 ms samples, 12.5 m traces
CH = (16, 48, 96, 192)        # the warm-start network's channels


def listed():
    return [
        # One small gather (256 samples, 64 traces, 8 velocities): an operator
        # pair inside a caller's own solver, where latency and launches count.
        dict(name="pair_small", kind="pair", B=1, nt=256, nx=64, nr=0, nv=8, nt0=1,
             wavelet=20.0, fmax=0.0, masked=False),
        # The receiver gathers of a survey, 64 at a time: 1024 samples, 256
        # traces, 32 velocities, 25 Hz wavelet.
        dict(name="pair_batch", kind="pair", B=64, nt=1024, nx=256, nr=0, nv=32, nt0=1,
             wavelet=25.0, fmax=0.0, masked=False),
        # Long, wide, odd-sized gathers (1500 samples, 417 traces) with dropped
        # traces and a band limit.
        dict(name="pair_ragged", kind="pair", B=5, nt=1500, nx=417, nr=0, nv=24, nt0=1,
             wavelet=0.0, fmax=80.0, masked=True),
        # Traces recorded off the regular grid (ch. 6: the trace transform
        # becomes a DFT at the trace positions).
        dict(name="pair_irregular", kind="pair", B=16, nt=1024, nx=256, nr=256, nv=32, nt0=1,
             wavelet=25.0, fmax=0.0, masked=False),
        # Robust deblending of one small gather, 5 x 20 iterations (a quick look
        # at one receiver).
        dict(name="deblend_small", kind="deblend", B=1, nt=256, nx=64, nv=8, wavelet=20.0,
             n_outer=5, n_cg=20, mu=0.0, masked=False, warm=False),
        # Robust deblending of a batch of full-size receiver gathers.
        dict(name="deblend_batch", kind="deblend", B=16, nt=1024, nx=256, nv=32, wavelet=25.0,
             n_outer=3, n_cg=10, mu=0.0, masked=False, warm=False),
        # A survey whose gathers have between 96 and 480 traces of 1500 samples.
        dict(name="batch_uneven", kind="batch", B=12, nt=1500, nx_lo=96, nx_hi=480, nv=24,
             wavelet=25.0, n_outer=3, n_cg=10),
        # AASHRT interpolation (24 velocities x 8 asymptote shifts) of gathers
        # with half of their traces missing.
        dict(name="fista_shifts", kind="fista", B=2, nt=1024, nx=128, nv=24, nt0=8, wavelet=25.0,
             n_iter=20, n_power=10),
        # The classical time-domain pair, to compare with or to check against.
        dict(name="td_pair", kind="td", B=8, nt=1024, nx=256, nv=32, nt0=1),
        # The learned warm start of 16 full-size gathers (24 velocity panels and
        # the residual weights).
        dict(name="predict_batch", kind="predict", B=16, nt=1024, nx=256, cout=25),
        # One training step of the warm start on the minibatch it is trained with.
        dict(name="train_step", kind="train", B=8, nt=1024, nx=256, cout=25),
        # Blending a cube of 256 shots x 64 receivers, cutting the shots back out
        # and sorting them to receiver gathers.
        dict(name="cube", kind="cube", ns=256, nr=64, nt=1024),
    ]


# ---------------------------------------------------------------------------
# drawn cases: the same kinds over the same ranges

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(n):
    p = 1
    while p < n:
        p *= 2
    return p


def _cells(B, nt, nx, P):
    """Padded spectrum cells of a batch (what the workspace and the work scale with)."""
    return B * P * (_pow2(2 * nx) // 2 + 1) * _pow2(2 * nt)


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "deblend", "deblend", "batch", "fista", "td",
                       "predict", "train", "cube"])
    if kind == "pair":
        c = dict(kind=kind, B=_log(rng, 1, 64), nt=_log(rng, 96, 1800), nx=_log(rng, 24, 480), nr=0,
                 nv=_log(rng, 4, 32), nt0=rng.choice([1, 1, 1, 4, 8]),
                 wavelet=rng.choice([0.0, 20.0, 25.0]), fmax=rng.choice([0.0, 0.0, 80.0]),
                 masked=rng.random() < 0.4)
        if rng.random() < 0.3:
            c["nr"] = max(8, int(c["nx"] * rng.uniform(0.5, 1.2)))
        while _cells(c["B"], c["nt"], c["nx"], c["nv"] * c["nt0"]) > 64 * 32 * 257 * 2048:
            c["B"] = max(1, c["B"] // 2)
            if c["B"] == 1:
                c["nt0"] = 1
        return c
    if kind == "deblend":
        c = dict(kind=kind, B=_log(rng, 1, 24), nt=_log(rng, 96, 1500), nx=_log(rng, 24, 320),
                 nv=_log(rng, 4, 32), wavelet=rng.choice([20.0, 25.0]),
                 n_outer=rng.randint(1, 3), n_cg=rng.randint(4, 10),
                 mu=rng.choice([0.0, 0.0, 0.0, 1e-3]), masked=rng.random() < 0.3,
                 warm=rng.random() < 0.3)
        while _cells(c["B"], c["nt"], c["nx"], c["nv"]) > 16 * 32 * 257 * 2048:
            c["B"] = max(1, c["B"] // 2)
        return c
    if kind == "batch":
        lo = _log(rng, 24, 120)
        return dict(kind=kind, B=rng.randint(3, 10), nt=_log(rng, 128, 1500), nx_lo=lo,
                    nx_hi=lo + _log(rng, 20, 300), nv=_log(rng, 4, 24), wavelet=25.0,
                    n_outer=rng.randint(1, 3), n_cg=rng.randint(4, 10))
    if kind == "fista":
        c = dict(kind=kind, B=_log(rng, 1, 8), nt=_log(rng, 96, 1200), nx=_log(rng, 24, 256),
                 nv=_log(rng, 4, 24), nt0=rng.choice([1, 4, 8]), wavelet=rng.choice([0.0, 25.0]),
                 n_iter=rng.randint(5, 20), n_power=rng.randint(5, 10))
        while _cells(c["B"], c["nt"], c["nx"], c["nv"] * c["nt0"]) > 2 * 192 * 129 * 2048:
            c["B"] = max(1, c["B"] // 2)
            if c["B"] == 1:
                c["nt0"] = 1
        return c
    if kind == "td":
        c = dict(kind=kind, B=_log(rng, 1, 16), nt=_log(rng, 64, 1600), nx=_log(rng, 12, 256),
                 nv=_log(rng, 1, 32), nt0=rng.choice([1, 1, 3]))
        while c["B"] * c["nv"] * c["nt0"] * c["nx"] ** 2 * c["nt"] > 8 * 32 * 256 ** 2 * 1024:
            if c["B"] > 1:
                c["B"] //= 2
            else:
                c["nx"] = max(12, c["nx"] // 2)
        return c
    if kind == "predict":
        return dict(kind=kind, B=_log(rng, 1, 16), nt=8 * _log(rng, 8, 128), nx=8 * _log(rng, 4, 32),
                    cout=rng.choice([9, 13, 25, 33]))
    if kind == "train":
        return dict(kind=kind, B=_log(rng, 1, 8), nt=8 * _log(rng, 8, 128), nx=8 * _log(rng, 4, 32),
                    cout=rng.choice([9, 13, 25, 33]))
    return dict(kind="cube", ns=_log(rng, 16, 256), nr=_log(rng, 4, 64), nt=_log(rng, 200, 1500))


# ---------------------------------------------------------------------------
# inputs

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed, salt=0):
    return torch.Generator(device=_dev()).manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _velocities(nv):
    return np.linspace(1400.0, 3500.0, nv).astype(np.float32)


def _t0s(nt0):
    return np.linspace(0.0, 0.4, nt0).astype(np.float32)


def _gathers(gen, B, nx, nt, fpeak=25.0, blended=True):
    """Gathers [B][nx][nt]: hyperbolic Ricker events and, when blended, two
    interfering sources whose traces carry random firing delays."""
    dev = _dev()
    T = nt * DT
    x = torch.arange(nx, device=dev)[None, :] * DX
    t = torch.arange(nt, device=dev)[None, None, :] * DT

    def u(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, device=dev, generator=gen)

    def source(n):
        d = torch.zeros((B, nx, nt), device=dev)
        for _ in range(n):
            tau, xa = u(0.05 * T, 0.8 * T, B, 1), u(0.0, (nx - 1) * DX, B, 1)
            v = u(1400.0, 3500.0, B, 1)
            amp = 1.0 + 0.3 * torch.randn((B, 1, 1), device=dev, generator=gen)
            tx = torch.sqrt(tau * tau + ((x - xa) / v) ** 2) + lag
            a = (math.pi * fpeak * (t - tx[:, :, None])) ** 2
            d += amp * (1.0 - 2.0 * a) * torch.exp(-a)
        return d

    lag = torch.zeros((B, nx), device=dev)
    d = source(10)
    if blended:
        for _ in range(2):
            lag = (u(0.0, 0.25 * T, B, nx) / DT).round() * DT
            d = d + u(1.0, 8.0, B, 1, 1) * source(6)
    return d.contiguous()


def _mask(gen, B, n, keep=0.5):
    m = (torch.rand((B, n), device=_dev(), generator=gen) < keep).float()
    m[:, 0] = 1.0
    return m


def _positions(seed, nx, nr):
    r = np.random.default_rng(seed)
    return np.sort(r.uniform(-0.45, nx - 0.55, nr)) * DX if nr != nx else \
        (np.arange(nx) + r.uniform(-0.45, 0.45, nx)) * DX


def _unet_params(seed, cout):
    r = np.random.default_rng(seed)
    out = []
    for ci, co, k in _layers(cout):
        out.append(r.standard_normal(co * ci * k * k, dtype=np.float32)
                   * np.float32(math.sqrt(2.0 / (ci * k * k))))
        out.append(np.float32(0.05) * r.standard_normal(co, dtype=np.float32))
    return np.concatenate(out)


def _layers(cout):
    c0, c1, c2, c3 = CH
    return [(1, c0, 3), (c0, c0, 3), (c0, c1, 3), (c1, c1, 3), (c1, c2, 3), (c2, c2, 3),
            (c2, c3, 3), (c3, c3, 3), (c3 + c2, c2, 3), (c2, c2, 3), (c2 + c1, c1, 3),
            (c1, c1, 3), (c1 + c0, c0, 3), (c0, c0, 3), (c0, cout, 1)]


def _batch_nx(c):
    """Trace counts of the survey's gathers."""
    r = np.random.default_rng([c["nt"], c["nx_lo"], c["nx_hi"]])
    return r.integers(c["nx_lo"], c["nx_hi"] + 1, size=c["B"])


def _inputs(c, seed):
    """What the calls read, by name."""
    g, dev, k = _gen(seed), _dev(), c["kind"]
    if k == "pair":
        P, nr = c["nv"] * c["nt0"], c["nr"] or c["nx"]
        return dict(m=torch.randn((c["B"], P, c["nx"], c["nt"]), device=dev, generator=g),
                    d=_gathers(g, c["B"], nr, c["nt"]),
                    mask=_mask(g, c["B"], nr) if c["masked"] else None)
    if k == "deblend":
        d = _gathers(g, c["B"], c["nx"], c["nt"])
        s = dict(d=d, mask=_mask(g, c["B"], c["nx"], 0.7) if c["masked"] else None, wr0=None)
        if c["warm"]:     # weights as a learned prediction gives them: smooth, of the data's size
            floor = 0.05 * d.abs().amax(dim=(1, 2), keepdim=True)
            s["wr0"] = torch.rsqrt(torch.maximum(d.abs(), floor)).contiguous()
        return s
    if k == "batch":
        nxs = _batch_nx(c)
        return dict(d=torch.cat([_gathers(g, 1, int(n), c["nt"]).reshape(-1) for n in nxs]))
    if k == "fista":
        d = _gathers(g, c["B"], c["nx"], c["nt"], blended=False)
        mask = _mask(g, c["B"], c["nx"])
        v0 = torch.randn((c["B"], c["nv"] * c["nt0"], c["nx"], c["nt"]), device=dev, generator=g)
        return dict(d=d, mask=mask, v0=v0)
    if k == "td":
        P = c["nv"] * c["nt0"]
        return dict(m=torch.randn((c["B"], P, c["nx"], c["nt"]), device=dev, generator=g),
                    d=_gathers(g, c["B"], c["nx"], c["nt"]))
    if k == "predict":
        return dict(x=_gathers(g, c["B"], c["nx"], c["nt"]))
    if k == "train":
        x = _gathers(g, c["B"], c["nx"], c["nt"])
        t = 0.3 * torch.randn((c["B"], c["cout"], c["nx"], c["nt"]), device=dev, generator=g)
        t[:, -1] += 0.5
        return dict(x=x, t=t)
    r = np.random.default_rng([int(seed), 7])
    fire = (np.arange(c["ns"]) * (c["nt"] // 2) + r.integers(0, max(1, c["nt"] // 4), c["ns"]))
    D = _gathers(g, c["ns"], c["nr"], c["nt"], blended=False)
    return dict(D=D, fire=torch.from_numpy(fire.astype(np.int32)).to(dev),
                nb=_record(c))


def _record(c):
    """Samples of the continuous record: shots fire every nt/2 samples, up to nt/4 late."""
    return (c["ns"] - 1) * (c["nt"] // 2) + c["nt"] // 4 + c["nt"]


def _lam(c):
    """Channel weights of the training loss: panels against residual weights."""
    P = c["cout"] - 1
    return np.array([0.25 / (P * 0.09)] * P + [0.75 / 0.09], np.float32)


class _State:
    def __init__(self, c, **kw):
        self.c = c
        self.__dict__.update(kw)


def prepare(case, seed):
    c, k, dev = dict(case), case["kind"], _dev()
    i = _inputs(c, seed)
    if k == "pair":
        plan = ashrt.Plan(c["nt"], c["nx"], DT, DX, _velocities(c["nv"]), t0s=_t0s(c["nt0"]),
                          wavelet_peak_hz=c["wavelet"], fmax_hz=c["fmax"], max_batch=c["B"],
                          trace_x=_positions(seed, c["nx"], c["nr"]) if c["nr"] else None)
        return _State(c, plan=plan, d_out=torch.empty_like(i["d"]), m_out=torch.empty_like(i["m"]),
                      **i)
    if k == "deblend":
        plan = ashrt.Plan(c["nt"], c["nx"], DT, DX, _velocities(c["nv"]), max_batch=c["B"],
                          wavelet_peak_hz=c["wavelet"], with_solver=True)
        return _State(c, plan=plan, drec=torch.empty_like(i["d"]),
                      m_out=torch.empty((c["B"],) + plan.model_shape, device=dev), **i)
    if k == "batch":
        b = ashrt.Batch(c["nt"], _batch_nx(c), DT, DX, _velocities(c["nv"]),
                        wavelet_peak_hz=c["wavelet"], with_solver=True)
        return _State(c, batch=b, m_out=torch.empty(b.model_elems, device=dev),
                      drec=torch.empty(b.data_elems, device=dev), **i)
    if k == "fista":
        plan = ashrt.Plan(c["nt"], c["nx"], DT, DX, _velocities(c["nv"]), t0s=_t0s(c["nt0"]),
                          max_batch=c["B"], wavelet_peak_hz=c["wavelet"], with_solver=True)
        return _State(c, plan=plan, drec=torch.empty_like(i["d"]), m_out=torch.empty_like(i["v0"]),
                      **i)
    if k == "td":
        return _State(c, v=_velocities(c["nv"]), t0s=_t0s(c["nt0"]), d_out=torch.empty_like(i["d"]),
                      m_out=torch.empty_like(i["m"]), **i)
    if k == "predict":
        net = ashrt.UNet(c["nx"], c["nt"], c["cout"], max_batch=c["B"],
                         params=_unet_params(seed, c["cout"]))
        return _State(c, net=net, wr0=torch.empty_like(i["x"]),
                      m0=torch.empty((c["B"], c["cout"] - 1, c["nx"], c["nt"]), device=dev), **i)
    if k == "train":
        net = ashrt.UNet(c["nx"], c["nt"], c["cout"], max_batch=c["B"],
                         params=_unet_params(seed, c["cout"]))
        return _State(c, net=net, lam=_lam(c), **i)
    return _State(c, rec=torch.empty((c["nr"], i["nb"]), device=dev), shots=torch.empty_like(i["D"]),
                  crg=torch.empty((c["nr"], c["ns"], c["nt"]), device=dev), **i)


def _misfits(reports):
    return np.array([r["misfit"] for r in reports], np.float32)


def run(s):
    c, k = s.c, s.c["kind"]
    if k == "pair":
        s.plan.forward(s.m, s.d_out, mask=s.mask, batch=c["B"])
        s.plan.adjoint(s.d, s.m_out, mask=s.mask, batch=c["B"])
        return {"d": s.d_out, "m": s.m_out}
    if k == "deblend":
        rep = s.plan.deblend(s.d, s.m_out, drec=s.drec, batch=c["B"], mask=s.mask, wr0=s.wr0,
                             n_outer=c["n_outer"], n_cg=c["n_cg"], mu=c["mu"])
        return {"m": s.m_out, "drec": s.drec, "misfit": _misfits(rep)}
    if k == "batch":
        rep = s.batch.deblend(s.d, s.m_out, drec=s.drec, n_outer=c["n_outer"], n_cg=c["n_cg"])
        return {"m": s.m_out, "drec": s.drec, "misfit": _misfits(rep)}
    if k == "fista":
        lf = s.plan.fista(s.d, s.m_out, s.v0, drec=s.drec, mask=s.mask, batch=c["B"], mu=0.01,
                          n_iter=c["n_iter"], n_power=c["n_power"])
        return {"m": s.m_out, "drec": s.drec, "lf": np.array(lf, np.float32)}
    if k == "td":
        ashrt.td_forward(c["nt"], c["nx"], DT, DX, s.v, s.m, s.d_out, t0s=s.t0s, batch=c["B"])
        ashrt.td_adjoint(c["nt"], c["nx"], DT, DX, s.v, s.d, s.m_out, t0s=s.t0s, batch=c["B"])
        return {"d": s.d_out, "m": s.m_out}
    if k == "predict":
        s.net.predict(s.x, s.m0, s.wr0)
        return {"m0": s.m0, "wr0": s.wr0}
    if k == "train":
        loss = s.net.train_step(s.x, s.t, 1e-4, channel_weight=s.lam)
        return {"loss": loss, "grads": s.net.grads()}
    ashrt.blend(s.D, s.fire, s.rec)
    ashrt.pseudo_deblend(s.rec, s.fire, s.shots)
    ashrt.sort_gathers(s.shots, s.crg)
    return {"record": s.rec, "shots": s.shots, "gathers": s.crg}


# ---------------------------------------------------------------------------
# what one pass cannot do without

def _pair_flops(nt, nx, P):
    """One operator pair of one gather: pruned 2-D transforms (5 N log2 N per
    complex length-N transform, half for real input) and the Stolt maps."""
    Nt, Nx = max(64, _pow2(2 * nt)), max(16, _pow2(2 * nx))
    Lh = Nx // 2 + 1
    return 2.0 * ((P + 1) * (nt * 2.5 * Nx * math.log2(Nx) + Lh * 5.0 * Nt * math.log2(Nt))
                  + 16.0 * P * Nt * Lh)


def _unet_flops(H, W, cout):
    div = [1, 1, 4, 4, 16, 16, 64, 64, 16, 16, 4, 4, 1, 1, 1]
    return sum(2.0 * ci * co * k * k * H * W / q for (ci, co, k), q in zip(_layers(cout), div))


def work(case):
    c, k = case, case["kind"]
    if k == "pair":
        P, nr = c["nv"] * c["nt0"], c["nr"] or c["nx"]
        return dict(bytes=8.0 * c["B"] * c["nt"] * (P * c["nx"] + nr),
                    flops=c["B"] * _pair_flops(c["nt"], c["nx"], P))
    if k == "deblend":
        pairs = c["n_outer"] * (c["n_cg"] + 0.5)
        return dict(bytes=4.0 * c["B"] * c["nt"] * c["nx"] * (c["nv"] + 2),
                    flops=c["B"] * pairs * _pair_flops(c["nt"], c["nx"], c["nv"]))
    if k == "batch":
        nxs = _batch_nx(c)
        pairs = c["n_outer"] * (c["n_cg"] + 0.5)
        return dict(bytes=4.0 * c["nt"] * float(nxs.sum()) * (c["nv"] + 2),
                    flops=sum(pairs * _pair_flops(c["nt"], int(n), c["nv"]) for n in nxs))
    if k == "fista":
        P = c["nv"] * c["nt0"]
        return dict(bytes=4.0 * c["B"] * c["nt"] * c["nx"] * (2 * P + 2),
                    flops=c["B"] * (c["n_iter"] + c["n_power"] + 0.5)
                    * _pair_flops(c["nt"], c["nx"], P))
    if k == "td":       # an interpolation (two multiply-adds) per sample, panel, apex and trace
        P = c["nv"] * c["nt0"]
        return dict(bytes=8.0 * c["B"] * c["nt"] * c["nx"] * (P + 1),
                    flops=8.0 * c["B"] * P * c["nx"] ** 2 * c["nt"])
    if k == "predict":
        n = c["B"] * c["nt"] * c["nx"]
        return dict(bytes=4.0 * n * (1 + c["cout"]),
                    flops=c["B"] * _unet_flops(c["nx"], c["nt"], c["cout"]))
    if k == "train":
        n = c["B"] * c["nt"] * c["nx"]
        return dict(bytes=4.0 * n * (1 + c["cout"]),
                    flops=3.0 * c["B"] * _unet_flops(c["nx"], c["nt"], c["cout"]))
    n = c["ns"] * c["nr"] * c["nt"]
    nb = _record(c)
    return dict(bytes=4.0 * (n + c["nr"] * nb) + 4.0 * (c["nr"] * nb + n) + 8.0 * n, flops=1.0 * n)


# ---------------------------------------------------------------------------
# the same numbers in FP64

class _Stolt:
    """The Stolt operator pair of one gather in FP64 on torch.fft."""

    def __init__(self, c, nx, positions=None):
        dev, f8 = _dev(), torch.float64
        self.nt, self.nx, self.nt0 = c["nt"], nx, c.get("nt0", 1)
        Nt, Nx = max(64, _pow2(2 * self.nt)), max(16, _pow2(2 * nx))
        self.Nt, self.Nx, Lh = Nt, Nx, Nx // 2 + 1
        k = torch.arange(Nt, device=dev, dtype=f8)
        k = torch.where(k <= Nt // 2, k, k - Nt)[None, :]
        self.taps = []
        for v in _velocities(c["nv"]).astype(np.float64):
            a = ((float(v) * torch.arange(Lh, device=dev, dtype=f8)) * float(Nt)) * DT / (float(Nx) * DX)
            a2 = (a * a)[:, None]
            ok = (k * k > a2) & (k != Nt // 2)
            u = torch.where(ok, torch.sign(k) * torch.sqrt(torch.clamp(k * k - a2, min=0.0)), 0.0 * k)
            f0 = torch.floor(u)
            i0 = torch.remainder(f0, Nt).long()
            i1 = torch.remainder(f0 + 1, Nt).long()
            w1 = torch.where(ok & (i1 != Nt // 2), u - f0, 0.0 * u)
            w0 = torch.where(ok & (i0 != Nt // 2), 1.0 - (u - f0), 0.0 * u)
            self.taps.append((i0, i1, w0, w1))
        f = (k[0].abs()) / (Nt * DT)
        W = torch.ones(Nt, device=dev, dtype=f8)
        if c["wavelet"] > 0:
            z = (f / c["wavelet"]) ** 2
            W = z * torch.exp(1.0 - z)
        if c.get("fmax", 0.0) > 0:
            W = torch.where(f > c["fmax"], 0.0 * W, W)
        W[Nt // 2] = 0.0
        self.W = W
        t0 = _t0s(self.nt0).astype(np.float64) if self.nt0 > 1 else np.zeros(1)
        self.phase = [torch.polar(torch.ones_like(W), -2.0 * math.pi * k[0] * float(t) / (Nt * DT))
                      for t in t0]
        self.E = None
        if positions is not None:
            x = torch.from_numpy(positions).to(dev)[:, None]
            l = torch.arange(Lh, device=dev, dtype=f8)[None, :]
            ph = torch.remainder(l * x / (Nx * DX), 1.0) * 2.0 * math.pi
            re, im = torch.cos(ph), torch.sin(ph)
            re[:, -1], im[:, -1] = torch.cos(math.pi * x[:, 0] / DX), 0.0
            cl = torch.full((1, Lh), 2.0, device=dev, dtype=f8)
            cl[0, 0] = cl[0, -1] = 1.0
            self.E = (re, im, cl)

    def forward(self, m, mask=None):
        """m [P][nx][nt] float64 (or float32, converted panel by panel) -> [nr][nt]."""
        D = 0.0
        nv = len(self.taps)
        for j, ph in enumerate(self.phase):
            Dj = 0.0
            for i, (i0, i1, w0, w1) in enumerate(self.taps):
                X = torch.fft.fft(torch.fft.rfft(m[j * nv + i].double(), n=self.Nx, dim=0), n=self.Nt,
                                  dim=1)
                Dj = Dj + w0 * X.gather(1, i0) + w1 * X.gather(1, i1)
            D = D + ph[None, :] * Dj
        Y = torch.fft.ifft(D * self.W[None, :], dim=1)[:, :self.nt]
        if self.E is None:
            d = torch.fft.irfft(Y, n=self.Nx, dim=0)[:self.nx]
        else:
            re, im, cl = self.E
            d = ((re * cl) @ Y.real.contiguous() - (im * cl) @ Y.imag.contiguous()) / self.Nx
        return d if mask is None else d * mask.double()[:, None]

    def adjoint(self, d, mask=None):
        """d [nr][nt] -> [P][nx][nt] float64."""
        d = d.double() if mask is None else d.double() * mask.double()[:, None]
        if self.E is None:
            Y = torch.fft.rfft(d, n=self.Nx, dim=0)
        else:
            re, im, _ = self.E
            Y = torch.complex(re.T @ d, -(im.T @ d))
        D = torch.fft.fft(Y, n=self.Nt, dim=1) * self.W[None, :]
        out = torch.empty((self.nt0 * len(self.taps), self.nx, self.nt), device=d.device,
                          dtype=torch.float64)
        nv = len(self.taps)
        for j, ph in enumerate(self.phase):
            Dj = D * ph.conj()[None, :]
            a, b = Dj.real.contiguous(), Dj.imag.contiguous()
            for i, (i0, i1, w0, w1) in enumerate(self.taps):
                re = torch.zeros_like(a).scatter_add_(1, i0, w0 * a).scatter_add_(1, i1, w1 * a)
                im = torch.zeros_like(b).scatter_add_(1, i0, w0 * b).scatter_add_(1, i1, w1 * b)
                M = torch.fft.ifft(torch.complex(re, im), dim=1)[:, :self.nt]
                out[j * nv + i] = torch.fft.irfft(M, n=self.Nx, dim=0)[:self.nx]
        return out


def _median(x):
    s = torch.sort(x).values
    n = s.numel()
    return 0.5 * (s[(n - 1) // 2] + s[n // 2])


def _irls(op, d, n_outer, n_cg, mu=0.0, mask=None, wr0=None):
    """IRLS / CGLS of one gather with p = q = 1 and the default options."""
    d = d.double()
    live = None if mask is None else mask.bool()
    dl = d if live is None else d * live[:, None]
    m, y, misfit = None, None, []
    for k in range(n_outer):
        if k == 0:
            Wr = torch.ones_like(d) if wr0 is None else wr0.double()
            Wi = 1.0
        else:
            r = d - y
            rl = (r if live is None else r[live]).reshape(-1)
            e = 1.345 * _median((rl - _median(rl)).abs()) / 0.6745
            r = r if live is None else r * live[:, None]
            Wr = torch.rsqrt(torch.maximum(r.abs(), e))
            Wi = torch.sqrt(torch.maximum(m.abs(), m.abs().max() / 100.0))

        def A(u):
            return Wr * op.forward(Wi * u, mask)

        def AT(r):
            return Wi * op.adjoint(Wr * r, mask)

        r = Wr * dl
        if k > 0:
            u = m / Wi
            r = r - (Wr * y if live is None else Wr * y * live[:, None])
        else:
            u = 0.0
        s = AT(r) - mu * u
        p = s.clone()
        gam = (s * s).sum()
        for it in range(n_cg):
            q = A(p)
            al = gam / ((q * q).sum() + mu * (p * p).sum())
            u = u + al * p
            if it + 1 == n_cg:
                break
            r = r - al * q
            s = AT(r) - mu * u
            g2 = (s * s).sum()
            p = s + (g2 / gam) * p
            gam = g2
        m = Wi * u
        y = op.forward(m)
        rr = d - y
        misfit.append(float((rr if live is None else rr[live]).abs().sum()))
    return m, y, misfit


def _fista(op, d, mask, v0, mu, n_iter, n_power):
    def normal(v):
        return op.adjoint(op.forward(v, mask), mask)

    v = v0.double()
    v = v / v.norm()
    for _ in range(n_power):
        w = normal(v)
        lam = w.norm()
        v = w / lam
    sd = d.double() * mask.double()[:, None]
    x = torch.zeros_like(v)
    y, t = x, 1.0
    for _ in range(n_iter):
        z = y - op.adjoint(op.forward(y, mask) - sd, mask) / lam
        xn = torch.sign(z) * torch.clamp(z.abs() - mu / (2.0 * lam), min=0.0)
        t1 = (1.0 + math.sqrt(1.0 + 4.0 * t * t)) / 2.0
        y = xn + ((t - 1.0) / t1) * (xn - x)
        x, t = xn, t1
    return x, op.forward(x), 2.0 * float(lam)


def _td_exact(c, i):
    nt, nx, B = c["nt"], c["nx"], c["B"]
    nv, t0s = c["nv"], _t0s(c["nt0"]).astype(np.float64)
    v = _velocities(nv).astype(np.float64)
    m, d = i["m"], i["d"].double()
    dev = d.device
    tau = torch.arange(nt, device=dev, dtype=torch.float64)
    dp = torch.zeros((B, nx, nt + 2), device=dev, dtype=torch.float64)   # samples >= nt drop here
    dpad = torch.cat([d, torch.zeros((B, nx, 2), device=dev, dtype=torch.float64)], 2)
    out = torch.zeros(m.shape, device=dev, dtype=torch.float64)
    for p in range(m.shape[1]):
        tj, vi = t0s[p // nv], v[p % nv]
        mp = m[:, p].double()
        for h in range(nx):
            s = tj / DT + torch.sqrt(tau * tau + (h * DX / (vi * DT)) ** 2)
            i0 = torch.floor(s)
            f = s - i0
            n = int((i0 < nt).sum())
            if n == 0:
                continue
            j0, f = i0[:n].long(), f[:n]
            for sg in ((1, -1) if h else (1,)):
                # apexes a and traces r = a + sg h
                ra, rr = (slice(0, nx - h), slice(h, nx)) if sg > 0 else (slice(h, nx), slice(0, nx - h))
                w = mp[:, ra, :n]
                dp[:, rr].index_add_(2, j0, (1.0 - f) * w)
                dp[:, rr].index_add_(2, j0 + 1, f * w)
                g = dpad[:, rr]
                out[:, p, ra, :n] += (1.0 - f) * g[:, :, j0] + f * g[:, :, j0 + 1]
    return {"d": dp[:, :, :nt].contiguous(), "m": out}


def _unet64(w, x, cout):
    """The network in FP64 on one image x [1][1][H][W] (already normalised)."""
    F = torch.nn.functional

    def cr(i, z):
        return F.relu(F.conv2d(z, w[2 * i], w[2 * i + 1], padding=1))

    s1 = cr(1, cr(0, x))
    s2 = cr(3, cr(2, F.avg_pool2d(s1, 2)))
    s3 = cr(5, cr(4, F.avg_pool2d(s2, 2)))
    b = cr(7, cr(6, F.avg_pool2d(s3, 2)))
    d3 = cr(9, cr(8, torch.cat([F.interpolate(b, scale_factor=2), s3], 1)))
    d2 = cr(11, cr(10, torch.cat([F.interpolate(d3, scale_factor=2), s2], 1)))
    d1 = cr(13, cr(12, torch.cat([F.interpolate(d2, scale_factor=2), s1], 1)))
    return F.conv2d(d1, w[28], w[29])


def _unet_weights(seed, cout):
    flat, out, o = torch.from_numpy(_unet_params(seed, cout)).to(_dev()).double(), [], 0
    for ci, co, k in _layers(cout):
        n = co * ci * k * k
        out += [flat[o:o + n].reshape(co, ci, k, k).clone(), flat[o + n:o + n + co].clone()]
        o += n + co
    return out


def _seconds(c):
    """About how long exact() takes, from the sizes."""
    k = c["kind"]
    if k == "td":
        P = c["nv"] * c["nt0"]
        return 2e-4 * 2 * P * c["nx"] + 1.5e-10 * c["B"] * P * c["nx"] ** 2 * c["nt"]
    if k in ("predict", "train"):
        n = 3 if k == "train" else 1
        return n * c["B"] * _unet_flops(c["nx"], c["nt"], c["cout"]) / 0.25e12
    if k == "cube":
        return 0.0
    P = c["nv"] * c.get("nt0", 1)
    nx = c["nx_hi"] if k == "batch" else c["nx"]
    n = {"pair": 1.0, "deblend": c.get("n_outer", 0) * (c.get("n_cg", 0) + 1.0),
         "batch": c.get("n_outer", 0) * (c.get("n_cg", 0) + 1.0),
         "fista": c.get("n_iter", 0) + c.get("n_power", 0) + 0.5}[k]
    return n * c["B"] * P * (4e-4 + 0.5e-9 * _pow2(2 * c["nt"]) * _pow2(2 * nx))


def exact(case, seed):
    c, k = dict(case), case["kind"]
    if _seconds(c) > 16.0:
        return None
    i = _inputs(c, seed)
    if k == "pair":
        op = _Stolt(c, c["nx"], _positions(seed, c["nx"], c["nr"]) if c["nr"] else None)
        ms = [None] * c["B"] if i["mask"] is None else list(i["mask"])
        d = torch.stack([op.forward(i["m"][b], ms[b]) for b in range(c["B"])])
        del i["m"]
        m = torch.empty((c["B"], c["nv"] * c["nt0"], c["nx"], c["nt"]), device=d.device,
                        dtype=torch.float64)
        for b in range(c["B"]):
            m[b] = op.adjoint(i["d"][b], ms[b])
        return {"d": d, "m": m}
    if k == "deblend":
        op = _Stolt(c, c["nx"])
        r = [_irls(op, i["d"][b], c["n_outer"], c["n_cg"], c["mu"],
                   None if i["mask"] is None else i["mask"][b],
                   None if i["wr0"] is None else i["wr0"][b]) for b in range(c["B"])]
        return {"m": torch.stack([x[0] for x in r]), "drec": torch.stack([x[1] for x in r]),
                "misfit": np.array([x[2] for x in r])}
    if k == "batch":
        r, o = [], 0
        for n in _batch_nx(c):
            d = i["d"][o:o + int(n) * c["nt"]].reshape(int(n), c["nt"])
            o += int(n) * c["nt"]
            r.append(_irls(_Stolt(c, int(n)), d, c["n_outer"], c["n_cg"]))
        return {"m": torch.cat([x[0].reshape(-1) for x in r]),
                "drec": torch.cat([x[1].reshape(-1) for x in r]),
                "misfit": np.array([x[2] for x in r])}
    if k == "fista":
        op = _Stolt(c, c["nx"])
        r = [_fista(op, i["d"][b], i["mask"][b], i["v0"][b], 0.01, c["n_iter"], c["n_power"])
             for b in range(c["B"])]
        return {"m": torch.stack([x[0] for x in r]), "drec": torch.stack([x[1] for x in r]),
                "lf": np.array([x[2] for x in r])}
    if k == "td":
        return _td_exact(c, i)
    if k in ("predict", "train"):
        w = _unet_weights(seed, c["cout"])
        x = i["x"].double()
        rms = x.square().mean(dim=(1, 2)).sqrt()
        if k == "predict":
            m0 = torch.empty((c["B"], c["cout"] - 1, c["nx"], c["nt"]), device=x.device,
                             dtype=torch.float64)
            wr0 = torch.empty_like(x)
            with torch.no_grad():
                for b in range(c["B"]):
                    y = _unet64(w, (x[b] / rms[b])[None, None], c["cout"])[0]
                    m0[b], wr0[b] = y[:-1] * rms[b], torch.exp(y[-1]) / torch.sqrt(rms[b])
            return {"m0": m0, "wr0": wr0}
        lam = torch.from_numpy(_lam(c)).to(x.device).double()[None, :, None, None]
        loss = 0.0
        for v in w:
            v.requires_grad_(True)
        for b in range(c["B"]):
            y = _unet64(w, (x[b] / rms[b])[None, None], c["cout"])
            e = (lam * (y - i["t"][b:b + 1].double()) ** 2).sum() / (c["B"] * c["nx"] * c["nt"])
            e.backward()
            loss += float(e)
        return {"loss": np.array(loss), "grads": torch.cat([v.grad.reshape(-1) for v in w])}
    D, fire = i["D"].double(), i["fire"].tolist()
    rec = torch.zeros((c["nr"], i["nb"]), device=D.device, dtype=torch.float64)
    for s, f in enumerate(fire):
        rec[:, f:f + c["nt"]] += D[s]
    shots = torch.stack([rec[:, f:f + c["nt"]] for f in fire])
    return {"record": rec, "shots": shots, "gathers": shots.transpose(0, 1).contiguous()}
