"""The projection's two forms (four samples a thread on aligned buffers, one
otherwise) give the same bits, also for pointing outside the map or the angle
table, which reads as zero and is reported for its detscan only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad_at", [(), (0,), (1, 2), (5, 1026, 4099), (4095, 4096, 5399)])
def test_forms_agree(bad_at):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(3)
    ndet, lens, nside = 1, (5400, 1024), 16
    off = np.array([0, 5400, 6424], np.int64)
    N, npix = 6424, 12 * nside * nside
    pix = rng.integers(0, npix, N).astype(np.int32)
    psi = rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(nside, ndet, len(lens), 32.5, off, tg.huff_encode(ndet, 2, off, pix),
                   tg.huff_encode(ndet, 2, off, psi))
    m = rng.standard_normal((npix, 4)).astype(np.float32)
    m[0] = np.nan                                   # a bad sample takes nothing from the first pixel
    pix[pix == 0] = 1
    for k, i in enumerate(bad_at):
        if k % 2:
            psi[i] = 4096
        else:
            pix[i] = (-1, npix, 2**31 - 1)[(k // 2) % 3]
    g = torch.tensor([1.5, 0.5], dtype=torch.float64, device="cuda")
    mt = torch.from_numpy(m).cuda()
    out = []
    for shift in (0, 1):
        p = torch.zeros(N + 8, dtype=torch.int32, device="cuda")[shift:shift + N]
        b = torch.zeros(N + 8, dtype=torch.int16, device="cuda")[shift:shift + N]
        s = torch.full((N + 8,), 7.0, dtype=torch.float32, device="cuda")
        p.copy_(torch.from_numpy(pix))
        b.copy_(torch.from_numpy(psi.astype(np.int16)))
        plan.project(mt, p, b, g, s[shift:])
        st = plan.status(raise_on_error=False)
        assert (st[0] != 0) == bool(bad_at) and st[1] == 0
        assert bool((s[shift + N:] == 7.0).all()) and bool((s[:shift] == 7.0).all())
        out.append(s[shift:shift + N].cpu().numpy())
    assert np.array_equal(out[0], out[1]) and np.isfinite(out[0]).all()
    assert (out[0][list(bad_at)] == 0.0).all()
    plan.close()
