"""The gap blocks' Toeplitz inverses at the edges of their range: one gap of
1, 2, 3, 511, 512 (the largest block), 513 and 700 samples (two blocks) per
detscan, under shallow and steep spectra.  With the block inverses alone the
CG's operator on a single block is the identity but for the detscan's ends
and the kernel's reference length, a few per cent: every iteration gains at
least a decade, so a residual of 1e-7 takes at most 8.  The draw itself is
the oracle's (relative l2 1e-5)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

SEED, BAND, IT = 23, 1, 2
LENGTHS = (1, 2, 3, 511, 512, 513, 700)


@pytest.mark.parametrize("fknee,alpha", [(0.02, -1.0), (0.2, -2.0), (1.0, -1.5)])
def test_single_gap_inverse(fknee, alpha):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    from gpu_workload import Workload
    cfg = synth.scaled(synth.CONFIGS["tiny"], nscan=len(LENGTHS), len_lo=15000, len_hi=20000, fsamp=78.8,
                       fknee_lo=fknee, fknee_hi=fknee, alpha_lo=alpha, alpha_hi=alpha)
    wl = Workload(cfg)
    f = np.zeros(wl.N, bool)
    for q, L in enumerate(LENGTHS):
        f[int(wl.off[q]) + 5000:int(wl.off[q]) + 5000 + L] = True
    flags = torch.from_numpy(tg.pack_flags(f).view(np.int32)).to(wl.dev)
    gain = torch.ones(wl.nq, dtype=torch.float64, device=wl.dev)
    x = torch.zeros(wl.N, dtype=torch.float32, device=wl.dev)
    its = torch.zeros(wl.nq, dtype=torch.int32, device=wl.dev)
    wl.plan.set_preconditioner(tg.PREC_BLOCKS)
    wl.plan.sample_ncorr(wl.t_d, wl.t_s, gain, flags, wl.t_psd, tg.Rng(SEED, BAND, IT), tg.MODE_DRAW, x, its,
                         cg_tol=1e-7)
    wl.plan.status()
    x, its = x.cpu().numpy().astype(np.float64), its.cpu().numpy()
    for q, L in enumerate(LENGTHS):
        sl = wl.sl(q)
        n = sl.stop - sl.start
        ref, _ = oracle.sample_ncorr(wl.d32[sl].astype(np.float64), wl.s32[sl].astype(np.float64), 1.0,
                                     (~f[sl]).astype(np.float64), *wl.band.psd[0], cfg.fsamp,
                                     oracle.omega1(SEED, BAND, q, IT, n), oracle.omega2(SEED, BAND, q, IT, n))
        assert np.linalg.norm(x[sl] - ref) < 1e-5 * np.linalg.norm(ref), (L, its[q])
        assert 1 <= its[q] <= 8, (L, its[q])


@pytest.mark.parametrize("length", [1024, 1030, 4096, 9000, 40000, 140000])
def test_kernel_of_every_detector(length):
    """Three detectors (one pair of a transform and one alone) of different
    spectra at reference lengths of two to three transform passes: each
    detector's own inverse serves its gap (the bound of the test above; under
    another detector's the CG takes tens of iterations)."""
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    from gpu_workload import Workload
    cfg = synth.scaled(synth.CONFIGS["tiny"], ndet=3, nscan=2, len_lo=length, len_hi=length, fsamp=78.8,
                       fknee_lo=0.02, fknee_hi=2.0, alpha_lo=-2.0, alpha_hi=-1.0, sigma0_jitter=0.2)
    wl = Workload(cfg)
    L = min(500, length // 10)
    f = np.zeros(wl.N, bool)
    for q in range(wl.nq):
        a = int(wl.off[q]) + length // 3
        f[a:a + L] = True
    flags = torch.from_numpy(tg.pack_flags(f).view(np.int32)).to(wl.dev)
    gain = torch.ones(wl.nq, dtype=torch.float64, device=wl.dev)
    x = torch.zeros(wl.N, dtype=torch.float32, device=wl.dev)
    its = torch.zeros(wl.nq, dtype=torch.int32, device=wl.dev)
    for levels in (tg.PREC_BLOCKS, tg.PREC_TWO_LEVEL):
        wl.plan.set_preconditioner(levels)
        wl.plan.sample_ncorr(wl.t_d, wl.t_s, gain, flags, wl.t_psd, tg.Rng(SEED, BAND, IT), tg.MODE_DRAW, x, its,
                             cg_tol=1e-7)
        wl.plan.status()
        assert 1 <= int(its.min()) and int(its.max()) <= 8, (levels, its.tolist())


def test_draw_on_other_streams_and_under_capture():
    """The draw's preparation runs beside its first passes on a stream of the
    plan: the same bits on the default stream, on another stream with the
    spectra freed in stream order right after the call, and replayed from a
    captured graph."""
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    from gpu_workload import Workload
    cfg = synth.scaled(synth.CONFIGS["tiny"], ndet=3, nscan=4, len_lo=9000, len_hi=20000, fsamp=78.8, flag_frac=0.03)
    wl = Workload(cfg)
    gain = torch.ones(wl.nq, dtype=torch.float64, device=wl.dev)
    out = [torch.zeros(wl.N, dtype=torch.float32, device=wl.dev) for _ in range(3)]

    def draw(psd, x):
        wl.plan.sample_ncorr(wl.t_d, wl.t_s, gain, wl.t_flags, psd, tg.Rng(SEED, BAND, IT), tg.MODE_DRAW, x)

    draw(wl.t_psd, out[0])
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        psd = wl.t_psd.clone()
        draw(psd, out[1])
        del psd
        torch.full((3, 3), float("nan"), dtype=torch.float64, device=wl.dev)      # may take the freed memory
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        draw(wl.t_psd, out[2])
    g.replay()
    torch.cuda.synchronize()
    wl.plan.status()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
