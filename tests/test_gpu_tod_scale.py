"""The decoded TOD is the FP64 product of count and scale, rounded once, for
scales over the whole range of FP64, among them those past FP32's: the same
bits as numpy's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SCALES = (1e-300, 1e-60, 1.4e-45, 1e-38, 1e-25, 3.3e-26, 1e-7, 1 / 3, 1.0, 2.0 ** -20, 1e20, 1e25, 1e38, 3.5e38,
          1e39, 1e300)


def test_scales_of_every_size():
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    rng = np.random.default_rng(8)
    n, nq = 4000, len(SCALES)
    off = np.arange(nq + 1, dtype=np.int64) * n
    N = nq * n
    z = tg.huff_encode(1, nq, off, np.zeros(N, np.int32))
    plan = tg.Plan(16, 1, nq, 32.5, off, z, z)
    counts = np.cumsum(rng.integers(-3, 4, N)).astype(np.int32)
    for q in range(nq):                              # zeros, small and large counts in every detscan
        counts[q * n:q * n + 40] = np.tile([0, 1, -1, 0, 3], 8)
        counts[q * n + 40:q * n + 80] = np.tile([2 ** 24 + 1, -2 ** 24 + 1, 2 ** 23 - 1, 0], 10)
    scale = np.array(SCALES)
    plan.attach_data(tg.huff_encode(1, nq, off, counts), scale, z, 1)
    d = torch.empty(N, device="cuda")
    flags = torch.empty((N + 31) // 32, dtype=torch.int32, device="cuda")
    plan.decode_data(d, flags)
    plan.status()
    with np.errstate(over="ignore", under="ignore"):
        want = (counts.astype(np.float64) * np.repeat(scale, n)).astype(np.float32)
    assert np.array_equal(d.cpu().numpy().view(np.int32), want.view(np.int32))
    plan.close()
