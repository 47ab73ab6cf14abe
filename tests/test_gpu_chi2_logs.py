"""The FP64 chi^2's sum of ln P, formed from products of four P, where P spans
more than half of FP64's range within a detscan: sigma0^2 near 1e-161 and a
slope of -90, so that products of two white-noise modes are subnormal while
those of two low modes are large.  No residual, so that the sum is all there
is; against the oracle's to 1e-11, the bound of the pass."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma0", [10.0 ** -80.8, 10.0 ** -80.5, 10.0 ** -79.9, 1e-60, 1e-3, 1.0])
@pytest.mark.parametrize("n", [2048, 8640])
def test_sum_of_logarithms(n, sigma0):
    torch = pytest.importorskip("torch")
    import paper_2201_03509_gb300 as tg
    psd = (sigma0, 14.0, -90.0 if n == 2048 else -70.0)
    off = np.array([0, n], np.int64)
    z = tg.huff_encode(1, 1, off, np.zeros(n, np.int32))
    plan = tg.Plan(16, 1, 1, 32.5, off, z, z)
    s = np.random.default_rng(1).standard_normal(n).astype(np.float32)
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    out = [torch.zeros(k, dtype=torch.float64, device="cuda") for k in (1, 1, 1, 3)]
    plan.chi2(t(s), t(s.astype(np.float64)), t(np.ones(1)), t(np.zeros((n + 31) // 32, np.int32)), t(np.array([psd])),
              *out, precision=plan.PREC_F64)
    plan.status()
    with np.errstate(all="ignore"):
        want = oracle.core.chi2_detscan(s.astype(np.float64), s.astype(np.float64), 1.0, np.ones(n), *psd, 32.5)["L"]
    assert np.isfinite(want)
    assert abs(float(out[0]) - want) <= 1e-11 * max(abs(want), n)
    plan.close()
