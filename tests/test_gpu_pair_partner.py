"""A detector's gap preconditioner does not depend on the detector that shares
its transform: three detectors (one pair and one alone), the second far
noisier, without finite noise, or with a spectrum far weaker than the first's.
Every detector of finite noise takes the CG iterations that it takes in a
band of its own (one more or less for the transform's rounding)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FSAMP = 78.8
PSD = np.array([[1.0e-3, 0.10, -1.5], [1.1e-3, 0.05, -1.8], [0.9e-3, 0.20, -1.2]])
PARTNER = {"alike": PSD[1], "1e3 louder": [1.1, 0.05, -1.8], "1e4 louder": [11.0, 0.05, -1.8],
           "1e4 quieter": [1.1e-7, 0.05, -1.8], "weak 1/f": [1.1e-3, 1e-5, -1.8], "infinite": [np.inf, 0.05, -1.8],
           "overflowing": [1e25, 0.05, -1.8], "no slope": [1.1e-3, 0.05, np.nan], "no knee": [1.1e-3, np.nan, -1.8]}


def _iterations(tg, torch, nscan, n, psd, d, f):
    nd = len(psd)
    off = np.arange(nd * nscan + 1, dtype=np.int64) * n
    rng = np.random.default_rng(5)
    pix, psi = rng.integers(0, 3072, off[-1]).astype(np.int32), rng.integers(0, 4096, off[-1]).astype(np.int32)
    plan = tg.Plan(16, nd, nscan, FSAMP, off, tg.huff_encode(nd, nscan, off, pix), tg.huff_encode(nd, nscan, off, psi))
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    x, its = torch.zeros(int(off[-1]), device="cuda"), torch.zeros(nd * nscan, dtype=torch.int32, device="cuda")
    gain = torch.ones(nd * nscan, dtype=torch.float64, device="cuda")
    out = []
    for levels in (tg.PREC_BLOCKS, tg.PREC_TWO_LEVEL):
        plan.set_preconditioner(levels)
        plan.sample_ncorr(t(d), torch.zeros_like(x), gain, t(tg.pack_flags(f).view(np.int32)), t(psd),
                          tg.Rng(1, 0, 0), tg.MODE_MEAN, x, its)
        status = plan.status(raise_on_error=False)
        out.append((its.cpu().numpy().reshape(nscan, nd), np.asarray(status).reshape(nscan, nd)))
    plan.close()
    return out


@pytest.mark.parametrize("n", [9000, 36000])
@pytest.mark.parametrize("partner", list(PARTNER))
def test_iterations_as_in_a_band_of_its_own(partner, n):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    nscan, psd = 2, PSD.copy()
    psd[1] = PARTNER[partner]
    rng = np.random.default_rng(7)
    d = np.empty((nscan, 3, n), np.float32)
    f = np.zeros((nscan, 3, n), bool)
    for s in range(nscan):
        for det in range(3):
            sig = psd[det, 0] if 0 < psd[det, 0] < 1e20 else 1.0
            drift = np.cumsum(rng.standard_normal(n))
            d[s, det] = sig * (rng.standard_normal(n) + drift / np.sqrt(n))
            for a in rng.integers(0, n - 300, 6):
                f[s, det, a:a + rng.integers(10, 300)] = True
    band = _iterations(tg, torch, nscan, n, psd, d.reshape(-1), f.reshape(-1))
    for det in range(3):
        if not (np.isfinite(psd[det]).all() and psd[det, 0] < 1e20):
            continue
        own = _iterations(tg, torch, nscan, n, psd[det:det + 1], d[:, det].reshape(-1), f[:, det].reshape(-1))
        for (a, sa), (b, sb) in zip(band, own):
            assert (sa[:, det] == 0).all() and (sb == 0).all(), partner
            assert (np.abs(a[:, det] - b[:, 0]) <= 1).all(), (partner, det, a[:, det], b[:, 0])
