"""The transform passes' pairs of columns and rows at their edges, through the
gain draw and the n_corr draw against the oracle: both factors of the split
even, one or both odd (a row without a partner, a column that is its own
mirror, a unit of two samples), powers of each radix, tiles of one pair and
ragged last tiles.  Tolerances are the draws' own: gain 1e-5 of its rms
(FP32 transforms), n_corr 1e-5 relative l2."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

SEED, BAND, IT = 29, 1, 3
# n = 2 m: m odd (675, 2187, 3125), small, prime powers, mixed
LENGTHS = (4, 6, 10, 18, 50, 1350, 4374, 6250, 2048, 8192, 10368, 30000, 36450)


@pytest.mark.parametrize("tile_pairs", [0, 1, 3, 64])
@pytest.mark.parametrize("mode", [0, 1])
def test_draws_at_every_parity(tile_pairs, mode):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(11)
    off = np.concatenate([[0], np.cumsum(LENGTHS)]).astype(np.int64)
    nq, N = len(LENGTHS), int(off[-1])
    pix = np.sort(rng.integers(0, 3072, N)).astype(np.int32)
    psi = rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(16, 1, nq, 32.5, off, tg.huff_encode(1, nq, off, pix), tg.huff_encode(1, nq, off, psi),
                   tile_pairs=tile_pairs)
    psd = np.array([[1e-3, 0.05, -1.5]])
    s = (1e-3 * rng.standard_normal(N)).astype(np.float32)       # of the noise: r = d - g s keeps FP32 accuracy
    d = (1.02 * s + 1e-3 * rng.standard_normal(N)).astype(np.float32)
    f = np.zeros(N, bool)
    for q, n in enumerate(LENGTHS):
        if n >= 1350 and q % 2:
            a = int(off[q]) + n // 3
            f[a:a + n // 60] = True
            f[off[q + 1] - 3:off[q + 1]] = True
    dev = "cuda:0"
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
    flags, gains = t(tg.pack_flags(f).view(np.int32)), [torch.zeros(nq, dtype=torch.float64, device=dev) for _ in range(3)]
    x = torch.zeros(N, dtype=torch.float32, device=dev)
    r = tg.Rng(SEED, BAND, IT)
    plan.sample_gain(t(d), t(s), flags, t(psd), r, mode, *gains)
    g_true = torch.full((nq,), 1.02, dtype=torch.float64, device=dev)
    plan.sample_ncorr(t(d), t(s), g_true, flags, t(psd), r, mode, x, cg_tol=1e-7)
    plan.status()
    g, mu, sig = (v.cpu().numpy() for v in gains)
    x = x.cpu().numpy().astype(np.float64)
    for q, n in enumerate(LENGTHS):
        sl = slice(int(off[q]), int(off[q + 1]))
        mask = (~f[sl]).astype(np.float64)
        P = oracle.core.noise_psd(n, 32.5, *psd[0])
        z = oracle.core.gain_normal(SEED, BAND, q, IT)
        ref = oracle.core.sample_gain(s[sl].astype(np.float64), d[sl].astype(np.float64), mask, P, z, mode)
        got = (g[q], mu[q], sig[q])
        for u, v in zip(got, ref):
            assert abs(u - v) <= 1e-5 * max(abs(ref[1]), ref[2]), (n, got, ref)
        w1 = oracle.omega1(SEED, BAND, q, IT, n) if mode == 0 else np.zeros(n)
        w2 = oracle.omega2(SEED, BAND, q, IT, n) if mode == 0 else np.zeros(n)
        want, _ = oracle.sample_ncorr(d[sl].astype(np.float64), s[sl].astype(np.float64), 1.02, mask, *psd[0], 32.5,
                                      w1, w2)
        assert np.linalg.norm(x[sl] - want) <= 1e-5 * np.linalg.norm(want), (n, tile_pairs)
    plan.close()
