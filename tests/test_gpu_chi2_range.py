"""The FP32 chi^2 over the whole range of its terms: detscans with terms of
ordinary size, past 1e18, past 3.4e38 once summed, and infinite ones, side by
side in one band.  What is finite is the FP64 oracle's (1e-6 of the value, or
of one a mode; gradients 1e-4 of their size: the bounds of the pass); a chi^2
with an infinite term is +inf, never NaN, and stays in its own detscan."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

FSAMP, PSD = 32.5, (1.0, 0.3, -0.6)
SIZES = (1.0, 1e6, 1e16, 1.5e18, 1e20, 1.0)          # data over sigma0: r^2 / P goes by the square


def _chi2(tg, torch, n, sel, pix, psi, d, s, f, gain):
    nq = len(sel)
    off = np.arange(nq + 1, dtype=np.int64) * n
    c = lambda v: np.concatenate([v[q * n:(q + 1) * n] for q in sel])  # noqa: E731
    plan = tg.Plan(16, 1, nq, FSAMP, off, tg.huff_encode(1, nq, off, c(pix)), tg.huff_encode(1, nq, off, c(psi)))
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    out = [torch.zeros(k, dtype=torch.float64, device="cuda") for k in (nq, nq, 1, 3)]
    plan.chi2(t(c(d)), t(c(s)), t(gain[sel]), t(tg.pack_flags(c(f)).view(np.int32)), t(np.array([PSD])), *out)
    plan.status()
    plan.close()
    return [o.cpu().numpy() for o in out]


@pytest.mark.parametrize("n", [4, 1024, 8640, 20000])
def test_terms_of_every_size(n):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    nq, N = len(SIZES), len(SIZES) * n
    rng = np.random.default_rng(3)
    pix, psi = rng.integers(0, 3072, N).astype(np.int32), rng.integers(0, 4096, N).astype(np.int32)
    s = (1 + 0.1 * rng.standard_normal(N)).astype(np.float32)
    d = (np.repeat(SIZES, n) * rng.standard_normal(N)).astype(np.float32)
    f = rng.random(N) < 0.03
    gain = np.full(nq, 1.1)
    ref = [oracle.core.chi2_detscan(d[q * n:(q + 1) * n].astype(np.float64), s[q * n:(q + 1) * n].astype(np.float64),
                                    gain[q], (~f[q * n:(q + 1) * n]).astype(np.float64), *PSD, FSAMP)
           for q in range(nq)]
    fin = [q for q in range(nq) if SIZES[q] < 1e19]
    L, dg, total, dpsd = _chi2(tg, torch, n, list(range(nq)), pix, psi, d, s, f, gain)
    assert not np.isnan(L).any()
    for q in fin:
        assert abs(L[q] - ref[q]["L"]) <= 1e-6 * max(abs(ref[q]["L"]), n), SIZES[q]
        assert abs(dg[q] - ref[q]["dg"]) <= 1e-4 * SIZES[q] * np.sqrt(n), SIZES[q]
    if n >= 1024:                                    # modes with r^2 / P past 3.4e38
        assert np.isposinf(L[[q for q in range(nq) if q not in fin]]).all() and np.isposinf(total[0])
    L, dg, total, dpsd = _chi2(tg, torch, n, fin, pix, psi, d, s, f, gain)
    want = np.sum([ref[q]["dpsd"] for q in fin], axis=0)
    assert total[0] == pytest.approx(sum(ref[q]["L"] for q in fin), rel=1e-6)
    assert np.abs(dpsd - want).max() <= 1e-4 * np.abs(want).max()
