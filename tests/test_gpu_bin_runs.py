"""Binning over runs of every kind against exact sums: single samples (a tile
of 2048 runs, 32 batches of staged outputs), runs around a quad's lanes and a
batch of 64, long ones, one longer than a tile, ragged mixtures, with samples
flagged.  Values to 1e-10 of the largest (the repository's bound
for FP64-accumulated maps; the products are exact and the sums FP32
double-words, 2^-44), hits exactly."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _pixels(kind, n, rng):
    if kind == "ragged":
        lens, pix = [], []
        while sum(lens) < n:
            lens.append(int(rng.choice([1, 2, 7, 8, 9, 15, 16, 17, 60, 300])))
        for i, L in enumerate(lens):
            pix += [i] * L
        return rng.permutation(np.array(pix[:n]))
    if kind == "in time":
        return np.arange(n) // 37
    return np.arange(n) % max(1, n // kind)          # runs of `kind` samples, interleaved


@pytest.mark.parametrize("kind", [1, 3, 4, 5, 8, 31, 32, 33, 60, 2048, 5000, "ragged", "in time"])
def test_runs_of_every_length(kind):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(7)
    ndet, lens, nside = 2, (5000, 2048, 6750), 64
    npix = 12 * nside * nside
    off = np.concatenate([[0], np.cumsum(np.repeat(lens, ndet))]).astype(np.int64)
    N, nq = int(off[-1]), ndet * len(lens)
    pix = np.concatenate([_pixels(kind, int(off[q + 1] - off[q]), rng) for q in range(nq)]).astype(np.int32)
    psi = rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(nside, ndet, len(lens), 32.5, off, tg.huff_encode(ndet, len(lens), off, pix),
                   tg.huff_encode(ndet, len(lens), off, psi))
    d = rng.standard_normal(N).astype(np.float32)
    x = (100.0 * rng.standard_normal(N)).astype(np.float32)
    f = rng.random(N) < 0.1
    psd = np.array([[1e-3, 0.05, -1.5], [2e-3, 0.05, -1.5]])
    gain = 1.0 + 0.1 * rng.standard_normal(nq)
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    A = torch.empty((npix, 6), dtype=torch.float64, device="cuda")
    b = torch.empty((npix, 3), dtype=torch.float64, device="cuda")
    hits = torch.empty(npix, dtype=torch.int32, device="cuda")
    plan.bin(t(psi.astype(np.int16)), t(d), t(x), t(gain), t(tg.pack_flags(f).view(np.int32)), t(psd), A, b, hits)
    plan.status()
    c, s = oracle.core.psi_trig_table()
    q = np.repeat(np.arange(nq), np.diff(off))
    w = (~f) / psd[q % ndet, 0] ** 2
    u = np.stack([np.ones(N), c[psi], s[psi]])
    r = d.astype(np.float64) - x.astype(np.float64)
    g = gain[q]
    for i, (k, l) in enumerate([(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]):
        ref = np.bincount(pix, w * g * g * u[k] * u[l], npix)
        assert np.abs(A[:, i].cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max(), (kind, i)
    for i in range(3):
        ref = np.bincount(pix, w * g * u[i] * r, npix)
        assert np.abs(b[:, i].cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max(), (kind, i)
    assert np.array_equal(hits.cpu().numpy(), np.bincount(pix[~f], minlength=npix))
    plan.close()
