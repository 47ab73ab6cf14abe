"""The scatter of the flagged samples' CG vector into the column tiles: single
flags at every place of a unit, at both ends and at the centre of a detscan,
for every parity of the transform's factors (a row that is its own mirror, a
column that is its own mirror, both), through the n_corr draw without a
preconditioner against the oracle (1e-5 relative l2, the draw's bound)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SEED, BAND, IT = 31, 2, 1
LENGTHS = (6, 10, 18, 30, 50, 64, 90, 150, 162, 250, 256, 450, 750, 1024, 1350, 2250, 4374, 6250, 8192, 12150)


@pytest.mark.parametrize("tile_pairs", [0, 1])
def test_flags_at_every_place(tile_pairs):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(19)
    off = np.concatenate([[0], np.cumsum(LENGTHS)]).astype(np.int64)
    nq, N = len(LENGTHS), int(off[-1])
    pix, psi = rng.integers(0, 3072, N).astype(np.int32), rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(16, 1, nq, 32.5, off, tg.huff_encode(1, nq, off, pix), tg.huff_encode(1, nq, off, psi),
                   tile_pairs=tile_pairs)
    psd = np.array([[1e-3, 0.05, -1.5]])
    s = (1e-3 * rng.standard_normal(N)).astype(np.float32)
    d = (1.02 * s + 1e-3 * rng.standard_normal(N)).astype(np.float32)
    f = rng.random(N) < 0.04
    for q, n in enumerate(LENGTHS):
        o, c = int(off[q]), n // 2
        f[[o, o + n - 1]] = True
        if n >= 18:
            f[o + c - 1:o + c + (1 if q % 2 else 2)] = True
        f[o + 2] = False
    dev = "cuda:0"
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
    x = torch.zeros(N, dtype=torch.float32, device=dev)
    gain = torch.full((nq,), 1.02, dtype=torch.float64, device=dev)
    plan.set_preconditioner(tg.PREC_NONE)
    plan.sample_ncorr(t(d), t(s), gain, t(tg.pack_flags(f).view(np.int32)), t(psd), tg.Rng(SEED, BAND, IT),
                      tg.MODE_DRAW, x, cg_tol=1e-7)
    plan.status()
    x = x.cpu().numpy().astype(np.float64)
    for q, n in enumerate(LENGTHS):
        sl = slice(int(off[q]), int(off[q + 1]))
        want, _ = oracle.sample_ncorr(d[sl].astype(np.float64), s[sl].astype(np.float64), 1.02,
                                      (~f[sl]).astype(np.float64), *psd[0], 32.5,
                                      oracle.omega1(SEED, BAND, q, IT, n), oracle.omega2(SEED, BAND, q, IT, n))
        assert np.linalg.norm(x[sl] - want) <= 1e-5 * np.linalg.norm(want), (n, tile_pairs)
    plan.close()
