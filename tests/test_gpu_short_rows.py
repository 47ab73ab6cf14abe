"""The row passes' distribution of a tile's rows over a CTA's warps: detscans
whose row transforms are far shorter than the CTA (several rows a step), about
a warp, and just past a power of two, with one and several rows a tile, through
the FP64 chi^2 (1e-11 of the value, or of one a mode; the gradients 1e-9 of
their size: the bounds of the pass) and the FP32 gain (1e-5 of its rms)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

LENGTHS = (4, 8, 12, 16, 24, 32, 60, 64, 90, 128, 160, 250, 256, 270, 486, 512, 640, 1000, 1024, 1080, 2048, 2250,
           4096, 4374, 5120, 8192, 16384, 16200)


@pytest.mark.parametrize("tile_pairs", [0, 1])
@pytest.mark.parametrize("max_radix", [0, 5])
def test_short_rows(tile_pairs, max_radix):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(17)
    off = np.concatenate([[0], np.cumsum(LENGTHS)]).astype(np.int64)
    nq, N = len(LENGTHS), int(off[-1])
    pix, psi = rng.integers(0, 3072, N).astype(np.int32), rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(16, 1, nq, 32.5, off, tg.huff_encode(1, nq, off, pix), tg.huff_encode(1, nq, off, psi),
                   tile_pairs=tile_pairs, max_radix=max_radix)
    psd = np.array([[1.1, 0.3, -1.2]])
    s = rng.standard_normal(N).astype(np.float32)
    d = (1.02 * s + rng.standard_normal(N)).astype(np.float32)
    f = rng.random(N) < 0.05
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    flags, gain = t(tg.pack_flags(f).view(np.int32)), np.full(nq, 0.97)
    out = [torch.zeros(k, dtype=torch.float64, device="cuda") for k in (nq, nq, 1, 3)]
    plan.chi2(t(d), t(s.astype(np.float64)), t(gain), flags, t(psd), *out, precision=plan.PREC_F64)
    g = [torch.zeros(nq, dtype=torch.float64, device="cuda") for _ in range(3)]
    plan.sample_gain(t(d), t(s), flags, t(psd), tg.Rng(1, 0, 0), tg.MODE_MEAN, *g)
    plan.status()
    L, dg, total, dpsd = (o.cpu().numpy() for o in out)
    mu, sig = g[1].cpu().numpy(), g[2].cpu().numpy()
    want = []
    for q, n in enumerate(LENGTHS):
        sl = slice(int(off[q]), int(off[q + 1]))
        m = (~f[sl]).astype(np.float64)
        r = oracle.core.chi2_detscan(d[sl].astype(np.float64), s[sl].astype(np.float64), gain[q], m, *psd[0], 32.5)
        want.append(r["dpsd"])
        assert abs(L[q] - r["L"]) <= 1e-11 * max(abs(r["L"]), n), n
        assert abs(dg[q] - r["dg"]) <= 1e-9 * max(abs(r["dg"]), np.sqrt(n)), n
        P = oracle.core.noise_psd(n, 32.5, *psd[0])
        _, rmu, rsig = oracle.core.sample_gain(s[sl].astype(np.float64), d[sl].astype(np.float64), m, P, 0.0, 1)
        assert abs(mu[q] - rmu) <= 1e-5 * max(abs(rmu), rsig) and abs(sig[q] - rsig) <= 1e-5 * rsig, n
    want = np.sum(want, axis=0)
    assert np.abs(dpsd - want).max() <= 1e-9 * np.abs(want).max()
    plan.close()
