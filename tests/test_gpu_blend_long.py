"""Blending, pseudo-deblending and sorting where rows are cut into pieces and where few
samples are blended: few long rows, rows on both sides of a piece, records of at most
128 samples (several receivers per CTA), lists of every length modulo the eight shots in
flight, the longest list.  The record is a float sum in shot order, compared bit for bit
with numpy; the copies are exact.  And a long row must not be left to one warp."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _blend_ref(D, fire, nb):
    ns, nr, nt = D.shape
    ref = np.zeros((nr, nb), np.float32)
    for i, f in enumerate(fire.astype(np.int64)):
        lo, hi = max(0, f), min(nb, f + nt)
        if lo < hi:
            ref[:, lo:hi] += D[i, :, lo - f:hi - f]
    return ref


@pytest.mark.parametrize("ns,nr,nt,nb", [
    (1, 1, 100003, 100003), (2, 1, 65536, 70000), (1, 3, 255, 257), (3, 2, 256, 512),
    (2, 2, 257, 255), (1, 1, 4096, 4096),          # pieces of a row
    (9, 17, 40, 1), (9, 17, 40, 31), (9, 9, 40, 32), (9, 9, 40, 33), (15, 5, 64, 64), (16, 5, 64, 65),
    (17, 3, 200, 128), (7, 3, 200, 129),           # receivers side by side
    (8192, 2, 5, 96), (8191, 1, 300, 300),         # the longest list
    (24, 1300, 50, 2000), (12, 350, 40, 7000),     # four samples per thread
])
def test_pieces_and_lists(lib, ns, nr, nt, nb):
    import torch
    from paper_1711_10214_gb300 import ashrt
    rng = np.random.default_rng(ns + nt)
    D = rng.standard_normal((ns, nr, nt)).astype(np.float32)
    fire = rng.integers(-nt // 2, max(1, nb - nt // 2), ns).astype(np.int32)
    Dd, fd = torch.from_numpy(D).cuda(), torch.from_numpy(fire).cuda()
    b = torch.full((nr, nb), float("nan"), device="cuda")
    ashrt.blend(Dd, fd, b)
    ref = _blend_ref(D, fire, nb)
    assert np.array_equal(b.cpu().numpy(), ref)
    shots = torch.full_like(Dd, float("nan"))
    ashrt.pseudo_deblend(b, fd, shots)
    want = np.zeros_like(D)
    for i, f in enumerate(fire.astype(np.int64)):
        lo, hi = max(0, f), min(nb, f + nt)
        if lo < hi:
            want[i, :, lo - f:hi - f] = ref[:, lo:hi]
    assert np.array_equal(shots.cpu().numpy(), want)
    for shift in (0, 1):
        src = torch.empty(D.size + 4, device="cuda")[shift:shift + D.size].view(ns, nr, nt)
        src.copy_(Dd)
        dst = torch.full((nr, ns, nt), float("nan"), device="cuda")
        ashrt.sort_gathers(src, dst)
        assert np.array_equal(dst.cpu().numpy(), D.transpose(1, 0, 2))


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


def test_long_rows_use_the_chip(lib):
    """Four rows of a million samples against 4000 rows of a thousand, the same bytes:
    within a factor of five (left to a warp per row they took 50 to 90 times as long)."""
    import torch
    from paper_1711_10214_gb300 import ashrt
    t = {}
    for ns, nr, nt in ((2, 2, 1000000), (2000, 2, 1000)):
        D = torch.randn((ns, nr, nt), device="cuda")
        out, srt = torch.empty_like(D), torch.empty((nr, ns, nt), device="cuda")
        fire = torch.arange(ns, device="cuda", dtype=torch.int32) * nt
        b = torch.randn((nr, ns * nt), device="cuda")
        t[ns] = (_best_us(lambda: ashrt.pseudo_deblend(b, fire, out)),
                 _best_us(lambda: ashrt.sort_gathers(D, srt)))
    for long_rows, short_rows in zip(t[2], t[2000]):
        assert long_rows <= 5.0 * short_rows, t
