"""Gaps cut anew when the Toeplitz tables stop short of the longest block: at
f_knee 10 Hz and slope -6 the recursion's pivots run out well below order 300
(an FP64 recursion on the kernel with FP32 rounding stops between 119 and 282),
so that no row past that order is written by the call.  The draws of a plan that
served a shallow spectrum before, whose tables still hold those rows, are those
of a new plan, bit for bit; a detscan whose cut passes 256 blocks goes without
a preconditioner."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FSAMP, N1 = 78.8, 16384
GAPS = ((1,), (100,), (300,), (465,), (511,), (512,), (513,), (700,), (250, -1, 250), (511, -1, 1, -1, 512),
        (40,) * 20, (5,) * 252 + (511,) * 4)          # -1: one sample between two gaps


def _flags():
    f = np.zeros((len(GAPS), N1), bool)
    for q, gaps in enumerate(GAPS):
        at = 100 + q
        for k, L in enumerate(gaps):
            if L < 0:
                continue
            f[q, at:at + L] = True
            at += L + (1 if k + 1 < len(gaps) and gaps[k + 1] < 0 else 25)
        assert at < N1
    return f.reshape(-1)


def _draw(plan, tg, torch, d, flags, psd, levels, maxit):
    N, nq = d.numel(), len(GAPS)
    x, its = torch.zeros(N, device="cuda"), torch.zeros(nq, dtype=torch.int32, device="cuda")
    plan.set_preconditioner(levels)
    plan.sample_ncorr(d, torch.zeros_like(x), torch.ones(nq, dtype=torch.float64, device="cuda"), flags,
                      torch.tensor([psd], dtype=torch.float64, device="cuda"), tg.Rng(4, 0, 1), tg.MODE_DRAW, x, its,
                      cg_maxiter=maxit)
    plan.status(raise_on_error=False)
    return x.cpu().numpy().reshape(nq, N1), its.cpu().numpy()


@pytest.mark.parametrize("alpha", [-4.0, -5.0, -6.0])
def test_cut_anew(alpha):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    nq = len(GAPS)
    off = np.arange(nq + 1, dtype=np.int64) * N1
    z = tg.huff_encode(1, nq, off, np.zeros(nq * N1, np.int32))
    rng = np.random.default_rng(2)
    d = torch.from_numpy((1e-3 * rng.standard_normal(nq * N1)).astype(np.float32)).cuda()
    flags = torch.from_numpy(tg.pack_flags(_flags()).view(np.int32)).cuda()
    steep, shallow = (1e-3, 10.0, alpha), (1e-3, 0.02, -1.0)
    plans = [tg.Plan(16, 1, nq, FSAMP, off, z, z) for _ in range(2)]
    _, its = _draw(plans[1], tg, torch, d, flags, shallow, tg.PREC_TWO_LEVEL, 500)
    assert (its[:-1] >= 1).all() and its.max() <= 20              # full tables there
    none, none_its = _draw(plans[0], tg, torch, d, flags, steep, tg.PREC_NONE, 40)
    for levels in (tg.PREC_BLOCKS, tg.PREC_TWO_LEVEL):
        (a, ia), (b, ib) = (_draw(p, tg, torch, d, flags, steep, levels, 40) for p in plans)
        assert np.array_equal(ia, ib) and np.array_equal(a.view(np.int32), b.view(np.int32))
        if alpha == -6.0:
            assert ia[-1] == none_its[-1] and np.array_equal(a[-1].view(np.int32), none[-1].view(np.int32))
    for p in plans:
        p.close()
