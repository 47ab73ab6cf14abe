"""Timing cases of the Gibbs TOD step: what a user of this framework runs,
through its public entry points (``Plan``, ``GibbsTODStep``, ``tod_chi2``).

A case is a slice of a band (detectors x pointing periods) or one layer of the
step on such a slice: the shapes are those of the bands this repository
configures (30, 44 and 70 GHz-like: sample rate, detectors, scan lengths,
Nside), with fewer scans than a whole mission so that the inputs are quick to
make; a process that holds one range of a band's scans runs exactly these.

Inputs are drawn on the GPU from the seed alone: a spinning scan strategy
(one revolution a minute, spin axis stepping from scan to scan), HEALPix RING
pixels, 4096 polarisation-angle bins, gains near one, 1/f plus white noise,
gaps of flagged samples.  ``exact`` computes the same outputs in FP64 with
torch and numpy alone (its own DCT, Philox streams, conjugate gradients).

The draws' results that are held in FP64 words but come from FP32 transforms
(gains, chi^2, log-likelihoods) are returned as the FP32 numbers that they
carry; what the library sums in FP64 (normal equations, maps, the FP64 chi^2)
is returned in FP64.
"""
import math
import random

import numpy as np
import torch

import paper_2201_03509_gb300 as tg
from paper_2201_03509_gb300.chi2 import tod_chi2
from paper_2201_03509_gb300.step import GibbsTODStep

BAND, ITERATION = 0, 3
F64, F32, I64, I32 = torch.float64, torch.float32, torch.int64, torch.int32
DEV = "cuda:0"
ADC_STEPS = 100.0               # ADC quanta per sigma0: about 9.2 bits a sample once coded
FLAG_EXCLUDE, FLAG_INFO, FLAG_SELECT = 2, 16, 0xF
PSD_STEPS, PSD_STEP = 10, 2e-4  # Metropolis steps of a call and their size (ln f_knee, alpha)
RCOND_STEP, RCOND_BIN = 1e-6, 1e-3


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def _case(name, kind, ndet, nscan, lo, hi, fsamp, nside, flagged=True, **options):
    return dict(name=name, kind=kind, ndet=ndet, nscan=nscan, len_lo=lo, len_hi=hi, fsamp=fsamp, nside=nside,
                flagged=flagged, **options)


def listed():
    return [
        # The smallest whole step (the tiny band: one detector, gap-free): a
        # sampler's unit of work when it is developed or run on a laptop-size
        # problem; launches and serial chains count.
        _case("step tiny", "step", 1, 16, 4096, 4096, 32.5, 16, flagged=False),
        # Whole steps of a scan range of the 30 and the 70 GHz bands: the
        # program's main loop on one process's share.
        _case("step 30GHz", "step", 4, 60, 90000, 140000, 32.5, 512),
        _case("step 70GHz", "step", 12, 36, 150000, 300000, 78.8, 1024),
        # The captured step on compressed data with the smooth gain prior: a
        # long chain replays one graph per iteration.
        _case("replay 30GHz", "replay", 4, 10, 90000, 140000, 32.5, 512),
        # The conditional mean on a few short, ragged detscans: gap filling of
        # a data selection, latency-bound.
        _case("ncorr mean short", "ncorr", 2, 5, 9001, 30011, 32.5, 512, mode="mean"),
        # The n_corr draw by itself at 44 and 70 GHz lengths: the layer that
        # takes two thirds of a step.
        _case("ncorr 44GHz", "ncorr", 6, 18, 136000, 204000, 46.5, 512, mode="draw"),
        _case("ncorr 70GHz", "ncorr", 12, 30, 150000, 300000, 78.8, 1024, mode="draw"),
        # The gain draw (forward and inverse transforms without a draw per mode).
        _case("gain 70GHz", "gain", 12, 30, 150000, 300000, 78.8, 1024),
        # chi^2 and its gradients for an optimiser over map, gains and noise:
        # forward and backward, in both precisions.
        _case("chi2 FP32", "chi2", 4, 200, 65536, 65536, 32.5, 256, flagged=False, fp64=False),
        _case("chi2 FP64", "chi2", 4, 25, 65536, 65536, 32.5, 256, flagged=False, fp64=True),
        # Map making from a cleaned timeline: binning and the per-pixel solve.
        _case("map 44GHz", "map", 6, 45, 136000, 204000, 46.5, 512),
        # Reading back compressed pointing, data and flags, then the noise-PSD
        # chain on a band's spectra.
        _case("decode and psd 30GHz", "decode", 4, 60, 90000, 140000, 32.5, 512),
    ]


def draw(rng: random.Random):
    """A slice or layer of the ranges above: 6e4 to 5e7 samples, scan
    lengths 4e3 to 3e5 (any raw length: the kept one is the FFT length)."""
    kind = rng.choice(["step", "step", "replay", "ncorr", "ncorr", "gain", "chi2", "map", "decode"])
    total = math.exp(rng.uniform(math.log(6e4), math.log(2.4e7 if kind in ("replay", "decode") else 5e7)))
    fsamp, nside = rng.choice([(32.5, 256), (32.5, 512), (46.5, 512), (78.8, 512), (78.8, 1024)])
    ndet = rng.choice([1, 2, 3, 4, 6, 7, 12])
    length = min(math.exp(rng.uniform(math.log(4001.0), math.log(3e5))), total / ndet)
    nscan = max(1, int(total / (ndet * length)))
    lo = max(1001, int(0.8 * length))
    case = dict(kind=kind, ndet=ndet, nscan=nscan, len_lo=lo, len_hi=max(lo, int(1.2 * length)), fsamp=fsamp,
                nside=nside, flagged=rng.random() < 0.8)
    if kind == "ncorr":
        case["mode"] = rng.choice(["draw", "draw", "mean"])
    if kind == "chi2":
        case["fp64"] = rng.random() < 0.3
        if case["fp64"]:
            case["nscan"] = max(1, nscan // 8)
    return case


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _fft_length(n):
    """The largest even 5-smooth number not above n."""
    best, a = 0, 2
    while a <= n:
        b = a
        while b <= n:
            c = b
            while c <= n:
                best = max(best, c)
                c *= 5
            b *= 3
        a *= 2
    return best


def _ang2pix_ring(nside, z, phi):
    """HEALPix RING pixel of (z = cos theta, phi in [0, 2 pi))."""
    za, tt = z.abs(), (phi * (2.0 / math.pi)).remainder(4.0)
    t1, t2 = nside * (0.5 + tt), nside * z * 0.75
    jp, jm = (t1 - t2).floor().to(I64), (t1 + t2).floor().to(I64)
    ir = nside + 1 + jp - jm
    ip = torch.div(jp + jm - nside + 2 - (ir & 1), 2, rounding_mode="floor").remainder(4 * nside)
    belt = 2 * nside * (nside - 1) + (ir - 1) * 4 * nside + ip
    tp, tmp = tt - tt.floor(), nside * torch.sqrt(3.0 * (1.0 - za))
    jp, jm = (tp * tmp).floor().to(I64), ((1.0 - tp) * tmp).floor().to(I64)
    ir = jp + jm + 1
    ip = (tt * ir).floor().to(I64).remainder(4 * ir)
    cap = torch.where(z > 0, 2 * ir * (ir - 1) + ip, 12 * nside * nside - 2 * ir * (ir + 1) + ip)
    return torch.where(za <= 2.0 / 3.0, belt, cap)


def _trig():
    """The tabulated cos 2psi, sin 2psi of the 4096 angle bins (FP32 values)."""
    psi = (np.arange(4096, dtype=np.float64) + 0.5) * (2.0 * math.pi / 4096)
    return (torch.from_numpy(np.cos(2 * psi).astype(np.float32)).to(DEV),
            torch.from_numpy(np.sin(2 * psi).astype(np.float32)).to(DEV))


class _Inputs:
    """The arrays of a case, on the GPU, concatenated in detscan order
    (q = scan * ndet + det)."""

    def __init__(self, case, seed):
        ndet, nscan, fs, nside = case["ndet"], case["nscan"], case["fsamp"], case["nside"]
        # the band's scan lengths belong to the case, everything else to the seed
        lengths = random.Random("%d %d %d" % (nscan, case["len_lo"], case["len_hi"]))
        self.n = [_fft_length(lengths.randint(case["len_lo"], case["len_hi"])) for _ in range(nscan)]
        host = random.Random(seed)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        self.off = np.zeros(nscan * ndet + 1, np.int64)
        self.off[1:] = np.cumsum(np.repeat(np.array(self.n, np.int64), ndet))
        N, npix = int(self.off[-1]), 12 * nside * nside
        self.N, self.npix, self.nq = N, npix, nscan * ndet

        def uniform(*shape, lo=0.0, hi=1.0):
            return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=F64)

        self.psd = torch.stack([uniform(ndet, lo=0.8e-3, hi=1.2e-3), uniform(ndet, lo=0.02, hi=0.2),
                                uniform(ndet, lo=-2.0, hi=-1.0)], 1)
        self.gain = 1.0 + 0.01 * torch.randn(self.nq, generator=g, device=DEV, dtype=F64)
        self.map = torch.zeros(npix, 4, device=DEV, dtype=F32)
        self.map[:, 0] = 1e-4 * torch.randn(npix, generator=g, device=DEV)
        self.map[:, 1:3] = 1e-5 * torch.randn(npix, 2, generator=g, device=DEV)
        self.pix = torch.empty(N, device=DEV, dtype=I32)
        self.psi = torch.empty(N, device=DEV, dtype=I32)
        self.d = torch.empty(N, device=DEV, dtype=F32)
        det = torch.arange(ndet, device=DEV, dtype=F64)[:, None]
        sa, ca = torch.sin(torch.deg2rad(85.0 + 0.35 * det)), torch.cos(torch.deg2rad(85.0 + 0.35 * det))
        cos2, sin2 = _trig()
        phase = [2 * math.pi * host.random() for _ in range(2 * nscan)]
        period = 60.0 if nside > 64 else 7.0
        step = 360.0 / 365.25 / 24.0 if nside > 64 else 112.5
        for s, n in enumerate(self.n):
            lam = math.radians(step * s)
            cl, sl = math.cos(lam), math.sin(lam)
            spin = (torch.arange(n, device=DEV, dtype=F64) * (2 * math.pi / (fs * period)) + phase[2 * s])[None, :] + 0.02 * det
            cs, sn = torch.cos(spin), torch.sin(spin)
            # axis (cl, sl, 0), perp = axis x z = (sl, -cl, 0), w = axis x perp = (0, 0, -1)
            x, y, z = ca * cl + sa * cs * sl, ca * sl - sa * cs * cl, (-sa * sn).clamp(-1.0, 1.0)
            dx, dy, dz = -sa * sn * sl, sa * sn * cl, -sa * cs
            phi = torch.atan2(y, x).remainder(2 * math.pi)
            st = torch.sqrt((1.0 - z * z).clamp_min(1e-30))
            sp, cp = torch.sin(phi), torch.cos(phi)
            ang = torch.atan2(-sp * dx + cp * dy, -z * cp * dx - z * sp * dy + st * dz)
            psi = (ang + torch.deg2rad(45.0 * det) + phase[2 * s + 1]).remainder(2 * math.pi)
            o = int(self.off[s * ndet])
            sl_ = slice(o, o + ndet * n)
            pix = _ang2pix_ring(nside, z, phi)
            psi = (psi * (4096 / (2 * math.pi))).to(I64).remainder(4096)
            self.pix[sl_], self.psi[sl_] = pix.to(I32).reshape(-1), psi.to(I32).reshape(-1)
            m = self.map[pix]
            sky = m[..., 0] + m[..., 1] * cos2[psi] + m[..., 2] * sin2[psi]
            # white noise plus 1/f noise with the detector's spectrum
            p = self.psd.to(F32)
            k = torch.arange(1, n // 2 + 1, device=DEV, dtype=F32)[None, :]
            amp = math.sqrt(n / 2) * p[:, :1] * (k * (fs / n) / p[:, 1:2]) ** (0.5 * p[:, 2:])
            spec = torch.zeros(ndet, n // 2 + 1, device=DEV, dtype=torch.complex64)
            spec[:, 1:] = amp * torch.complex(*torch.randn(2, ndet, n // 2, generator=g, device=DEV))
            noise = torch.fft.irfft(spec, n) + p[:, :1] * torch.randn(ndet, n, generator=g, device=DEV)
            gq = self.gain[s * ndet:(s + 1) * ndet, None].to(F32)
            self.d[sl_] = (gq * sky + noise).reshape(-1)
        # flagged gaps of 10..500 samples, about 2 % of each detscan
        self.flagged = torch.zeros(N, device=DEV, dtype=torch.bool)
        if case["flagged"]:
            edge = torch.zeros(N + 1, device=DEV, dtype=I32)
            nq_len = torch.from_numpy(np.diff(self.off)).to(DEV)
            hi = (nq_len // 50).clamp(11, 500)
            count = ((0.02 * nq_len) / (0.5 * (10 + hi))).ceil().to(I64)
            q = torch.repeat_interleave(torch.arange(self.nq, device=DEV), count)
            n_q, o_q = nq_len[q], torch.from_numpy(self.off).to(DEV)[q]
            a = (uniform(len(q)) * n_q).to(I64).minimum(n_q - 1)
            b = torch.minimum(a + 10 + (uniform(len(q)) * (hi[q] - 9)).to(I64), n_q)
            one = torch.ones(len(q), device=DEV, dtype=I32)
            edge.index_add_(0, o_q + a, one)
            edge.index_add_(0, o_q + b, -one)
            self.flagged = edge[:N].cumsum(0, dtype=I32) > 0
        # quality words: the excluding bit on the gaps, an informational bit elsewhere
        info = (torch.arange(N, device=DEV) // 1777).remainder(23) == int(seed) % 23
        self.flag_words = (self.flagged.to(I32) * FLAG_EXCLUDE + info.to(I32) * FLAG_INFO)
        self.scale = (self.psd[:, 0] / ADC_STEPS).repeat(nscan)
        self.nlen = torch.from_numpy(np.diff(self.off)).to(DEV)
        self.generator = g

    def counts(self):
        """The detector data as ADC counts of sigma0 / 100."""
        return torch.round(self.d.to(F64) / torch.repeat_interleave(self.scale, self.nlen)).to(I32)

    def spectrum(self, case):
        """DCT spectra of n_corr draws: Gaussian modes of the 1/f prior."""
        k = torch.cat([torch.arange(n, device=DEV, dtype=F32).repeat(case["ndet"]) for n in self.n])
        q = torch.repeat_interleave(torch.arange(self.nq, device=DEV), self.nlen)
        p = self.psd.to(F32)[q % case["ndet"]]
        f = k * (case["fsamp"] / 2) / self.nlen[q]
        amp = torch.where(k > 0, p[:, 0] * (f.clamp_min(1e-9) / p[:, 1]) ** (0.5 * p[:, 2]), torch.zeros_like(k))
        return amp * torch.randn(self.N, generator=self.generator, device=DEV)

    def unit_signal(self):
        """s = P m at unit gain, FP32 (what a projection leaves)."""
        cos2, sin2 = _trig()
        m, b = self.map[self.pix], self.psi.to(I64)
        return m[:, 0] + m[:, 1] * cos2[b] + m[:, 2] * sin2[b]


def _plan(case, x):
    nd, ns = case["ndet"], case["nscan"]
    return tg.Plan(case["nside"], nd, ns, case["fsamp"], x.off,
                   tg.huff_encode(nd, ns, x.off, x.pix.cpu().numpy()),
                   tg.huff_encode(nd, ns, x.off, x.psi.cpu().numpy()))


def _attach(case, x, plan):
    nd, ns = case["ndet"], case["nscan"]
    plan.attach_data(tg.huff_encode(nd, ns, x.off, x.counts().cpu().numpy()), x.scale.cpu().numpy(),
                     tg.huff_encode(nd, ns, x.off, x.flag_words.cpu().numpy()), FLAG_SELECT)


def _packed(x):
    return tg.pack_flags(x.flagged.cpu().numpy())


def _words(x):
    return torch.from_numpy(_packed(x).view(np.int32)).to(DEV)


def _gain_prior(case):
    return np.tile([1e-3, -2.0], (case["ndet"], 1))


def _parameters(case, x):
    """A point on an optimiser's way: the true map, gains a per cent off, noise
    parameters not yet fitted; leaves of the graph in the pass's precision."""
    t = F64 if case["fp64"] else F32
    psd = x.psd * torch.tensor([1.1, 1.3, 0.9], device=DEV, dtype=F64)
    return [v.detach().to(t).clone().requires_grad_(True) for v in (x.map[:, :3], x.gain * 1.01, psd)]


def prepare(case, seed):
    kind, x = case["kind"], _Inputs(case, seed)
    plan = _plan(case, x)
    s = dict(kind=kind, plan=plan, rng=tg.Rng(seed, BAND, ITERATION))
    if kind in ("step", "replay"):
        if kind == "replay":
            _attach(case, x, plan)
            s["step"] = GibbsTODStep(plan, x.psd.cpu().numpy(), None, rcond_min=RCOND_STEP, data_streams=True,
                                     gain_prior=_gain_prior(case))
        else:
            s["step"] = GibbsTODStep(plan, x.psd.cpu().numpy(), _packed(x), rcond_min=RCOND_STEP)
            s["step"].set_tod(x.d)
        s["map"] = x.map
        if kind == "replay":
            s["step"].capture(x.map, seed, BAND)
        return s
    s.update(psd=x.psd, flags=_words(x), d=x.d)
    empty = lambda *shape, dtype=F32: torch.empty(*shape, device=DEV, dtype=dtype)  # noqa: E731
    if kind == "ncorr":
        s.update(mode=tg.MODE_MEAN if case["mode"] == "mean" else tg.MODE_DRAW, s=x.unit_signal(), gain=x.gain,
                 ncorr=empty(x.N))
    elif kind == "gain":
        s.update(s=x.unit_signal(), out=[empty(x.nq, dtype=F64) for _ in range(3)])
    elif kind == "chi2":
        s.update(parameters=_parameters(case, x), precision=plan.PREC_F64 if case["fp64"] else plan.PREC_F32)
    elif kind == "map":
        # the timeline's correlated part, as a draw would have left it
        ncorr = 0.5 * x.d
        s.update(psi=x.psi.to(torch.int16), ncorr=ncorr, gain=x.gain, A=empty(x.npix, 6, dtype=F64),
                 b=empty(x.npix, 3, dtype=F64), hits=empty(x.npix, dtype=I32), map=empty(3, x.npix, dtype=F64),
                 map32=empty(x.npix, 4), rcond=empty(x.npix, dtype=F64), valid=empty(x.npix, dtype=torch.uint8))
    elif kind == "decode":
        _attach(case, x, plan)
        nd = case["ndet"]
        s.update(pix=empty(x.N, dtype=I32), psi=empty(x.N, dtype=torch.int16), d=empty(x.N),
                 flags=empty((x.N + 31) // 32, dtype=I32), spec=x.spectrum(case), psd_out=empty(nd, 3, dtype=F64),
                 accepted=empty(nd, dtype=I32), loglike=empty(nd, dtype=F64))
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------

def run(s):
    kind, plan = s["kind"], s["plan"]
    if kind in ("step", "replay"):
        st = s["step"]
        if kind == "step":
            st.run(s["map"], s["rng"])
        else:
            st.replay(ITERATION)
        return dict(map=st.map32, ncorr=st.ncorr, gain=st.gain.to(F32), hits=st.hits, valid=st.valid)
    if kind == "ncorr":
        plan.sample_ncorr(s["d"], s["s"], s["gain"], s["flags"], s["psd"], s["rng"], s["mode"], s["ncorr"])
        return s["ncorr"]
    if kind == "gain":
        plan.sample_gain(s["d"], s["s"], s["flags"], s["psd"], s["rng"], tg.MODE_DRAW, *s["out"])
        return dict(zip(("gain", "mean", "rms"), torch.stack(s["out"]).to(F32)))
    if kind == "chi2":
        m, g, p = s["parameters"]
        value = tod_chi2(m, g, p, plan, s["d"], s["flags"], s["precision"])
        grads = torch.autograd.grad(value, [m, g, p])
        return dict(value=value.detach().to(m.dtype), map=grads[0], gain=grads[1], psd=grads[2])
    if kind == "map":
        plan.bin(s["psi"], s["d"], s["ncorr"], s["gain"], s["flags"], s["psd"], s["A"], s["b"], s["hits"])
        plan.solve_maps(s["A"], s["b"], s["hits"], RCOND_BIN, s["map"], s["map32"], s["rcond"], s["valid"])
        return {k: s[k] for k in ("A", "b", "hits", "map", "map32", "valid")}
    plan.decode(s["pix"], s["psi"])
    plan.decode_data(s["d"], s["flags"])
    plan.sample_noise_psd(s["spec"], s["psd"], s["rng"], PSD_STEPS, PSD_STEP, PSD_STEP, s["psd_out"], s["accepted"],
                          s["loglike"])
    return dict(pix=s["pix"], psi=s["psi"], d=s["d"], flags=s["flags"], psd=s["psd_out"], accepted=s["accepted"],
                loglike=s["loglike"].to(F32))


def work(case):
    """Compulsory bytes (inputs once, outputs once; compressed pointing taken
    as one byte a sample, compressed data and flags as 1.3) and the arithmetic
    of the transforms (2.5 n log2 n each) and sums."""
    length = 0.5 * (case["len_lo"] + case["len_hi"])
    N = case["ndet"] * case["nscan"] * length
    npix = 12.0 * case["nside"] ** 2
    dct = 2.5 * N * math.log2(length)
    flag = 0.125
    if case["kind"] in ("step", "replay"):
        data = 1.3 if case["kind"] == "replay" else 4 + flag
        # gain: two forward transforms; n_corr: forward and back, and once more for the gaps
        return dict(bytes=N * (1 + data + 4) + npix * (16 + 16 + 8 * 3 + 4 + 1),
                    flops=dct * (4 + (2 if case["flagged"] else 0)) + 60 * N)
    if case["kind"] == "ncorr":
        return dict(bytes=N * (12 + flag), flops=dct * (4 if case["flagged"] else 2) + 10 * N)
    if case["kind"] == "gain":
        return dict(bytes=N * (8 + flag), flops=2 * dct + 10 * N)
    if case["kind"] == "chi2":
        w = 8 if case["fp64"] else 4
        return dict(bytes=N * (1 + 4 + flag) + npix * 6 * w, flops=2 * dct + 40 * N)
    if case["kind"] == "map":
        return dict(bytes=N * (10 + flag) + npix * (72 + 24 + 16 + 8 + 5), flops=30 * N + 60 * npix)
    # decode and the noise-PSD chain: one reading of the spectra per evaluation
    return dict(bytes=N * (2.3 + 6 + 4 + flag) + 4.0 * N * (PSD_STEPS + 1), flops=10.0 * N * (PSD_STEPS + 1))


# ----------------------------------------------------------------------------
# the same in FP64
# ----------------------------------------------------------------------------

def _dct(x):
    """Orthonormal DCT-II of the rows of x (even length)."""
    n = x.shape[1]
    v = torch.cat([x[:, ::2], x[:, 1::2].flip(1)], 1)
    k = torch.arange(n // 2 + 1, device=x.device, dtype=F64)
    y = torch.fft.rfft(v) * torch.polar(torch.full_like(k, math.sqrt(2.0 / n)), -math.pi * k / (2 * n))
    out = torch.cat([y.real, -y.imag[:, 1:n // 2].flip(1)], 1)
    out[:, 0] *= math.sqrt(0.5)
    return out


def _idct(X):
    n = X.shape[1]
    c = X * math.sqrt(n / 2.0)
    c[:, 0] *= math.sqrt(2.0)
    h = n // 2
    k = torch.arange(h + 1, device=X.device, dtype=F64)
    im = torch.zeros_like(c[:, :h + 1])
    im[:, 1:] = -c[:, h:].flip(1)
    v = torch.fft.irfft(torch.complex(c[:, :h + 1], im) * torch.polar(torch.ones_like(k), math.pi * k / (2 * n)), n)
    x = torch.empty_like(X)
    x[:, ::2], x[:, 1::2] = v[:, :h], v[:, h:].flip(1)
    return x


def _philox(seed, block, q, purpose, words):
    """Raw words of the Philox4x64 stream (q, purpose, iteration) from a block on."""
    counter = (ITERATION << 192 | purpose << 128 | q << 64 | block) - 1
    return np.random.Philox(key=seed | BAND << 64, counter=counter % (1 << 256)).random_raw(words)


def _normals(seed, q, purpose, n):
    """The first n normals of a timeline stream: Box-Muller pairs of 23-bit uniforms."""
    h = torch.from_numpy(_philox(seed, 0, q, purpose, 4 * (-(-n // 8))).view("<u4").astype(np.int64)).to(DEV)
    u = ((h >> 9).to(F64) + 0.5) * 2.0 ** -23
    r, a = torch.sqrt(-2.0 * torch.log(u[::2])), 2 * math.pi * u[1::2]
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], 1).reshape(-1)[:n]


def _uniform53(word):
    return ((int(word) >> 11) + 0.5) * 2.0 ** -53


def _cos_normal(w0, w1):
    return math.sqrt(-2.0 * math.log(_uniform53(w0))) * math.cos(2 * math.pi * _uniform53(w1))


class _Exact:
    """FP64 restatement of the step's layers on a case's inputs, scan by scan."""

    def __init__(self, case, seed, x=None):
        self.case, self.seed, self.x = case, seed, x or _Inputs(case, seed)
        self.cos2, self.sin2 = (v.to(F64) for v in _trig())

    def scans(self):
        nd = self.case["ndet"]
        for s, n in enumerate(self.x.n):
            o = int(self.x.off[s * nd])
            yield s * nd, n, slice(o, o + nd * n)

    def rows(self, v, sl):
        return v[sl].reshape(self.case["ndet"], -1).to(F64)

    def angles(self):
        b = self.x.psi.to(I64)
        return self.cos2[b], self.sin2[b]

    def signal(self, m):
        c, s = self.angles()
        p = self.x.pix.to(I64)
        return m[p, 0].to(F64) + m[p, 1].to(F64) * c + m[p, 2].to(F64) * s

    def noise(self, n, psd):
        f = torch.arange(n, device=DEV, dtype=F64)[None, :] * (self.case["fsamp"] / (2.0 * n))
        w = torch.zeros(psd.shape[0], n, device=DEV, dtype=F64)
        w[:, 1:] = (f[:, 1:] / psd[:, 1:2]) ** psd[:, 2:]
        return w                                            # (f / f_knee)^alpha, 0 at mode 0

    def gains(self, d, s, prior=None):
        nd, x = self.case["ndet"], self.x
        mu, sg = torch.empty(x.nq, device=DEV, dtype=F64), torch.empty(x.nq, device=DEV, dtype=F64)
        for q0, n, sl in self.scans():
            M = (~self.rows(x.flagged, sl).bool()).to(F64)
            P = x.psd[:, :1] ** 2 * (1.0 + self.noise(n, x.psd))
            sh, dh = _dct(M * self.rows(s, sl))[:, 1:], _dct(M * self.rows(d, sl))[:, 1:]
            a = (sh * sh / P[:, 1:]).sum(1)
            mu[q0:q0 + nd], sg[q0:q0 + nd] = (sh * dh / P[:, 1:]).sum(1) / a, a.rsqrt()
        if prior is None:
            z = torch.tensor([_cos_normal(*_philox(self.seed, 0, q, 0, 2)) for q in range(x.nq)], device=DEV, dtype=F64)
            return mu + z * sg, mu, sg
        # joint draw of each detector's scans under the smooth prior
        S, g = self.case["nscan"], torch.empty_like(mu)
        C = _dct(torch.eye(S, device=DEV, dtype=F64)).T if S > 1 and S % 2 == 0 else _cosines(S)
        for det in range(nd):
            sigma_g, alpha_g = prior[det]
            lam = torch.zeros(S, device=DEV, dtype=F64)
            lam[1:] = 1.0 / (sigma_g ** 2 * torch.arange(1, S, device=DEV, dtype=F64) ** alpha_g)
            a = 1.0 / sg[det::nd] ** 2
            w = [_philox(self.seed, s, det, 4, 4) for s in range(S)]
            w1 = torch.tensor([_cos_normal(v[0], v[1]) for v in w], device=DEV, dtype=F64)
            w2 = torch.tensor([_cos_normal(v[2], v[3]) for v in w], device=DEV, dtype=F64)
            rhs = a * mu[det::nd] + a.sqrt() * w1 + C.T @ (lam.sqrt() * w2)
            g[det::nd] = torch.linalg.solve(torch.diag(a) + C.T @ (lam[:, None] * C), rhs)
        return g, mu, sg

    def ncorr(self, d, s, gain, drawn=True):
        nd, x = self.case["ndet"], self.x
        out = torch.empty(x.N, device=DEV, dtype=F64)
        for q0, n, sl in self.scans():
            F = self.rows(x.flagged, sl)
            M, s2 = 1.0 - F, x.psd[:, :1] ** 2
            r = self.noise(n, x.psd)
            r[:, 1:] = 1.0 / r[:, 1:]
            beta, gamma = s2 / (1.0 + r), s2 * r / (1.0 + r)
            v = (self.rows(d, sl) - gain[q0:q0 + nd, None] * self.rows(s, sl)) / s2
            prior = 0.0
            if drawn:
                z1 = torch.stack([_normals(self.seed, q, 1, n) for q in range(q0, q0 + nd)])
                z2 = torch.stack([_normals(self.seed, q, 2, n) for q in range(q0, q0 + nd)])
                t = torch.arange(n, device=DEV)
                v = v + z1[:, torch.where(t % 2 == 0, t // 2, n - 1 - (t - 1) // 2)] / s2.sqrt()
                mode = torch.where(t < n // 2, 2 * t, 2 * (n - t) + 1)
                mode[0], mode[n // 2] = 0, 1
                prior = (r / s2).sqrt() * z2[:, mode]
            x0 = _idct(beta * (_dct(M * v) + prior))
            # the flagged samples: conjugate gradients on E^T C^T gamma C E y = E^T x0
            y, res = torch.zeros_like(x0), F * x0
            p, rr = res.clone(), (res * res).sum(1, keepdim=True)
            stop = 1e-24 * rr
            for _ in range(1000):
                if bool((rr <= stop).all()):
                    break
                Sp = F * _idct(gamma * _dct(p))
                a = torch.where(rr > stop, rr / (p * Sp).sum(1, keepdim=True), torch.zeros_like(rr))
                y, res = y + a * p, res - a * Sp
                new = (res * res).sum(1, keepdim=True)
                p = torch.where(rr > stop, res + new / rr.clamp_min(1e-300) * p, p)
                rr = torch.where(rr > stop, new, rr)
            out[sl] = (x0 + _idct(beta * _dct(y))).reshape(-1)
        return out

    def normal_equations(self, d, x_, gain):
        x, nd = self.x, self.case["ndet"]
        c, s = self.angles()
        keep = ~x.flagged
        q = torch.repeat_interleave(torch.arange(x.nq, device=DEV), x.nlen)[keep]
        p, c, s = x.pix.to(I64)[keep], c[keep], s[keep]
        g, s2 = gain[q], x.psd[q % nd, 0] ** 2
        wA, wb = g * g / s2, g / s2 * (d.to(F64) - x_.to(F64))[keep]
        total = lambda v: torch.zeros(x.npix, device=DEV, dtype=F64).index_add_(0, p, v)  # noqa: E731
        A = torch.stack([total(wA * v) for v in (torch.ones_like(c), c, s, c * c, c * s, s * s)], 1)
        b = torch.stack([total(wb * v) for v in (torch.ones_like(c), c, s)], 1)
        return A, b, total(torch.ones_like(c))

    @staticmethod
    def solve(A, b, hits, rcond_min):
        a00, a01, a02, a11, a12, a22 = A.unbind(1)
        det = a00 * (a11 * a22 - a12 * a12) - a01 * (a01 * a22 - a12 * a02) + a02 * (a01 * a12 - a11 * a02)
        dp = a00 * a11 * a22
        ok = (hits >= 3) & (dp > 0) & (det >= rcond_min * dp)
        full = torch.stack([a00, a01, a02, a01, a11, a12, a02, a12, a22], 1).reshape(-1, 3, 3)[ok]
        out = torch.zeros_like(b)
        scale = full.diagonal(dim1=1, dim2=2).rsqrt()
        L = torch.linalg.cholesky(full * scale[:, :, None] * scale[:, None, :])
        out[ok] = torch.cholesky_solve((b[ok] * scale)[:, :, None], L)[:, :, 0] * scale
        return out

    def chi2(self, m, gain, psd):
        x, nd = self.x, self.case["ndet"]
        s, v_all = self.signal(m), torch.empty(x.N, device=DEV, dtype=F64)
        value, dg, dp = 0.0, torch.empty(x.nq, device=DEV, dtype=F64), torch.zeros(nd, 3, device=DEV, dtype=F64)
        s0, fk, al = psd[:, :1], psd[:, 1:2], psd[:, 2:]
        for q0, n, sl in self.scans():
            M = 1.0 - self.rows(x.flagged, sl)
            sr, g = self.rows(s, sl), gain[q0:q0 + nd, None]
            rh = _dct(M * (self.rows(x.d, sl) - g * sr))
            w = self.noise(n, psd)
            P = s0 ** 2 * (1.0 + w)
            rh[:, 0] = 0.0
            value = value + 0.5 * (rh[:, 1:] ** 2 / P[:, 1:] + P[:, 1:].log()).sum()
            h = 0.5 * (1.0 / P - rh ** 2 / P ** 2)[:, 1:]
            f = torch.arange(1, n, device=DEV, dtype=F64) * (self.case["fsamp"] / (2.0 * n))
            dp += torch.stack([(h * 2 * P[:, 1:] / s0).sum(1), (h * (-s0 ** 2 * al * w[:, 1:] / fk)).sum(1),
                               (h * s0 ** 2 * w[:, 1:] * torch.log(f / fk)).sum(1)], 1)
            v = M * _idct(rh / P)
            dg[q0:q0 + nd] = -(M * sr * v).sum(1)
            v_all[sl] = (g * v).reshape(-1)
        c, sn = self.angles()
        p = x.pix.to(I64)
        dm = torch.stack([torch.zeros(x.npix, device=DEV, dtype=F64).index_add_(0, p, v_all * u)
                          for u in (torch.ones_like(c), c, sn)], 1)
        return dict(value=value, map=-dm, gain=dg, psd=dp)

    def psd_chain(self, spec):
        """The Metropolis chain on (ln f_knee, alpha) of every detector."""
        x, nd, fs = self.x, self.case["ndet"], self.case["fsamp"]
        state, loglike = x.psd.clone(), torch.empty(nd, device=DEV, dtype=F64)
        for det in range(nd):
            power, lnf = [], []
            for q0, n, sl in self.scans():
                power.append(self.rows(spec, sl)[det, 1:] ** 2)
                lnf.append(torch.log(torch.arange(1, n, device=DEV, dtype=F64) * (fs / (2.0 * n))))
            power, lnf = torch.cat(power), torch.cat(lnf)
            s0 = float(x.psd[det, 0])
            def value(lk, al):  # noqa: E306
                return -0.5 * float((power * torch.exp(-al * (lnf - lk)) / s0 ** 2 + 2 * math.log(s0) + al * (lnf - lk)).sum())
            lk, al = math.log(float(x.psd[det, 1])), float(x.psd[det, 2])
            cur = value(lk, al)
            for step in range(PSD_STEPS):
                w = _philox(self.seed, step, det, 3, 3)
                r, a = math.sqrt(-2 * math.log(_uniform53(w[0]))), 2 * math.pi * _uniform53(w[1])
                pk, pa = lk + PSD_STEP * r * math.cos(a), al + PSD_STEP * r * math.sin(a)
                if not (math.log(1e-4) <= pk <= math.log(10.0) and -4.0 <= pa <= -0.25):
                    continue
                new = value(pk, pa)
                if math.log(_uniform53(w[2])) < new - cur:
                    lk, al, cur = pk, pa, new
            if (lk, al) != (math.log(float(x.psd[det, 1])), float(x.psd[det, 2])):
                state[det, 1], state[det, 2] = math.exp(lk), al
            loglike[det] = cur
        return state, loglike


def _cosines(n):
    """The orthonormal DCT-II matrix of any length."""
    k = torch.arange(n, device=DEV, dtype=F64)
    C = torch.cos(math.pi * k[:, None] * (k[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
    C[0] *= math.sqrt(0.5)
    return C


def exact(case, seed):
    kind, e = case["kind"], _Exact(case, seed)
    x = e.x
    if kind in ("step", "replay"):
        d = x.d
        if kind == "replay":
            d = (x.counts().to(F64) * torch.repeat_interleave(x.scale, x.nlen)).to(F32)
        s = e.signal(x.map)
        gain, _, _ = e.gains(d, s, _gain_prior(case) if kind == "replay" else None)
        ncorr = e.ncorr(d, s, gain)
        A, b, hits = e.normal_equations(d, ncorr, gain)
        m = torch.zeros(x.npix, 4, device=DEV, dtype=F64)
        m[:, :3] = e.solve(A, b, hits, RCOND_STEP)
        return dict(map=m, ncorr=ncorr, gain=gain, hits=None, valid=None)
    if kind == "ncorr":
        return e.ncorr(x.d, x.unit_signal(), x.gain, case["mode"] == "draw")
    if kind == "gain":
        return dict(zip(("gain", "mean", "rms"), e.gains(x.d, x.unit_signal())))
    if kind == "chi2":
        m, g, p = (v.detach().to(F64) for v in _parameters(case, x))
        return e.chi2(m, g, p)
    if kind == "map":
        A, b, hits = e.normal_equations(x.d, 0.5 * x.d, x.gain)
        m = e.solve(A, b, hits, RCOND_BIN)
        m4 = torch.zeros(x.npix, 4, device=DEV, dtype=F64)
        m4[:, :3] = m
        return dict(A=A, b=b, hits=None, map=m.T.contiguous(), map32=m4, valid=None)
    d = x.counts().to(F64) * torch.repeat_interleave(x.scale, x.nlen)
    state, loglike = e.psd_chain(x.spectrum(case))
    return dict(pix=None, psi=None, d=d, flags=None, psd=state, accepted=None, loglike=loglike)
