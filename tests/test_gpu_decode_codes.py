"""Decoding of every kind of code, exactly: one symbol, codes within the
table, codes longer than it, more symbols than are staged in shared memory;
detscans below, at and just past a checkpoint block, and outputs at the start
of an allocation and one element into it (stores one by one)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pixels(kind, n, npix, rng):
    if kind == "one symbol":
        return np.full(n, 17)
    if kind == "table":
        return np.cumsum(rng.integers(-20, 21, n)) % npix
    if kind == "long codes":                        # geometric: a few symbols take most samples
        step = (rng.geometric(0.02, n) ** 2) * rng.choice([-1, 1], n)
        return np.cumsum(step) % npix
    return rng.integers(0, npix, n)                 # "many symbols": nearly every difference its own


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind", ["one symbol", "table", "long codes", "many symbols"])
def test_codes_of_every_kind(kind, shift):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(11)
    ndet, lens, nside = 2, (500, 512, 540, 1024, 20000), 512
    off = np.concatenate([[0], np.cumsum(np.repeat(lens, ndet))]).astype(np.int64)
    N, nq = int(off[-1]), ndet * len(lens)
    pix = np.concatenate([_pixels(kind, int(off[q + 1] - off[q]), 12 * nside * nside, rng)
                          for q in range(nq)]).astype(np.int32)
    psi = rng.integers(0, 4096, N).astype(np.int32)
    plan = tg.Plan(nside, ndet, len(lens), 32.5, off, tg.huff_encode(ndet, len(lens), off, pix),
                   tg.huff_encode(ndet, len(lens), off, psi))
    pix_out = torch.full((N + 2,), -1, dtype=torch.int32, device="cuda")
    psi_out = torch.full((N + 2,), -1, dtype=torch.int16, device="cuda")
    plan.decode(pix_out[shift:], psi_out[shift:])
    plan.status()
    assert np.array_equal(pix_out[shift:shift + N].cpu().numpy(), pix)
    assert np.array_equal(psi_out[shift:shift + N].cpu().numpy().astype(np.int32), psi)
    for out in (pix_out, psi_out):                  # nothing written around the outputs
        assert int((out[:shift] != -1).sum()) == 0 and int((out[shift + N:] != -1).sum()) == 0
    plan.close()
