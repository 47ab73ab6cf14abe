"""An n_corr draw whose preparation fails leaves nothing behind on the plan's
side stream: the caller's stream waits for what was queued, so a capture of the
failed call ends without a loose branch, and the plan serves the next call.
The failure is on the host alone: an error of an earlier call (a plan on a
device that does not exist) that the preparation's launch check picks up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_failed_preparation_is_joined():
    torch = pytest.importorskip("torch")
    import synth
    import paper_2201_03509_gb300 as tg
    from gpu_workload import Workload
    wl = Workload(synth.scaled(synth.CONFIGS["tiny"], ndet=2, nscan=3, len_lo=4000, len_hi=6000, flag_frac=0.03))
    gain = torch.ones(wl.nq, dtype=torch.float64, device=wl.dev)
    out = [torch.zeros(wl.N, dtype=torch.float32, device=wl.dev) for _ in range(2)]

    def draw(x):
        wl.plan.sample_ncorr(wl.t_d, wl.t_s, gain, wl.t_flags, wl.t_psd, tg.Rng(3, 0, 1), tg.MODE_DRAW, x)

    draw(out[0])
    torch.cuda.synchronize()
    off = np.array([0, 1024], np.int64)
    pix = tg.huff_encode(1, 1, off, np.zeros(1024, np.int32))
    g = torch.cuda.CUDAGraph()
    failed = False
    with torch.cuda.graph(g):                       # raises on a branch that is not joined
        out[1].fill_(7.0)
        with pytest.raises(tg.TodError):
            tg.Plan(16, 1, 1, 32.5, off, pix, pix, device=torch.cuda.device_count() + 98)
        try:
            draw(out[1])
        except tg.TodError:
            failed = True
    assert failed
    g.replay()
    torch.cuda.synchronize()
    assert bool((out[1] == 7.0).all())
    draw(out[1])
    torch.cuda.synchronize()
    wl.plan.status()
    assert torch.equal(out[0], out[1])
