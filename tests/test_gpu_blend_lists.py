"""Blending with the per-tile shot lists and the row copies at their edges: shots
in any order, many passes over the shots, shots that reach no tile, receivers
sharing a list, rows with and without 16-byte alignment.  The record is a float
sum in shot order, so it is compared bit for bit with the same sum in numpy; the
copies are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nr,nt,nb", [
    (1, 1, 1, 1), (300, 3, 37, 1025), (700, 2, 40, 5000), (257, 9, 3000, 1024),
    (40, 60, 16, 1024 * 170),                 # four receivers per CTA
])
def test_blend_and_copies(lib, ns, nr, nt, nb):
    import torch
    from paper_1711_10214_gb300 import ashrt
    rng = np.random.default_rng(ns + nt)
    D = rng.standard_normal((ns, nr, nt)).astype(np.float32)
    fire = rng.integers(-nt - 5, nb + 5, ns).astype(np.int32)
    if ns > 3:
        fire[:3] = (-2 ** 31, 2 ** 31 - 1, 0)
    ref = np.zeros((nr, nb), np.float32)
    for i, f in enumerate(fire.astype(np.int64)):
        lo, hi = max(0, f), min(nb, f + nt)
        if lo < hi:
            ref[:, lo:hi] += D[i, :, lo - f:hi - f]
    Dd, fd = torch.from_numpy(D).cuda(), torch.from_numpy(fire).cuda()
    b = torch.full((nr, nb), np.nan, device="cuda")
    ashrt.blend(Dd, fd, b)
    assert np.array_equal(b.cpu().numpy(), ref)
    shots = torch.full_like(Dd, np.nan)
    ashrt.pseudo_deblend(b, fd, shots)
    want = np.zeros_like(D)
    for i, f in enumerate(fire.astype(np.int64)):
        lo, hi = max(0, f), min(nb, f + nt)
        if lo < hi:
            want[i, :, lo - f:hi - f] = ref[:, lo:hi]
    assert np.array_equal(shots.cpu().numpy(), want)
    # sorting, on a 16-byte boundary and four bytes behind it
    for shift in (0, 1):
        src = torch.empty(D.size + 4, device="cuda")[shift:shift + D.size].view(ns, nr, nt)
        src.copy_(Dd)
        dst = torch.full((nr, ns, nt), np.nan, device="cuda")
        ashrt.sort_gathers(src, dst)
        assert np.array_equal(dst.cpu().numpy(), D.transpose(1, 0, 2))
