"""A band of more detscans than a launch has CTAs, most of them one tile, some
long, some without flags: the n_corr draw's passes over the list of iterating
detscans, as launches and in the cooperative tail, give the bits and the
iteration counts of the same kernels launched once per detscan."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", ["PREC_NONE", "PREC_TWO_LEVEL"])
def test_lists_of_many_detscans(levels):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(23)
    ndet = 3
    lens = [int(tg.fft_length(int(v))) for v in rng.integers(600, 2500, 330)]
    for i in (0, 57, 200, 329):
        lens[i] = 40000
    off = np.concatenate([[0], np.cumsum(np.repeat(lens, ndet))]).astype(np.int64)
    nscan, nq, N = len(lens), ndet * len(lens), int(off[-1])
    z = np.zeros(N, np.int32)
    plan = tg.Plan(16, ndet, nscan, 78.8, off, tg.huff_encode(ndet, nscan, off, z), tg.huff_encode(ndet, nscan, off, z))
    plan.set_preconditioner(getattr(tg, levels))
    f = np.zeros(N, bool)
    for q in range(nq):
        if q % 11 == 5:
            continue                                 # no flags: never on the list
        n = int(off[q + 1] - off[q])
        for a in rng.integers(0, n - 30, max(1, n // 600)):
            f[off[q] + a:off[q] + a + rng.integers(2, 30)] = True
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    d, flags = t((1e-3 * rng.standard_normal(N)).astype(np.float32)), t(tg.pack_flags(f).view(np.int32))
    psd = t(np.array([[1e-3, 0.1, -1.5], [1.1e-3, 0.5, -1.9], [0.9e-3, 0.02, -1.1]]))
    gain = torch.ones(nq, dtype=torch.float64, device="cuda")
    out = []
    for schedule in (plan.SCHED_PERSISTENT, plan.SCHED_PER_SCAN):
        plan.set_schedule(schedule)
        x, its = torch.zeros(N, device="cuda"), torch.zeros(nq, dtype=torch.int32, device="cuda")
        plan.sample_ncorr(d, torch.zeros_like(x), gain, flags, psd, tg.Rng(2, 0, 4), tg.MODE_DRAW, x, its)
        plan.status()
        out.append((x, its))
    assert int(out[0][1].max()) > 3                  # past the launched iterations
    assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][0], out[1][0])
    plan.close()
