"""Standardised scores are the correctly rounded quotients (score - mean) / SD of
the statistics that are returned, whatever the scores' scale: the kernel
multiplies by the bin's reciprocal and corrects the product, and divides where
the quotient or the numerator leaves the ordinary range.  Marker counts around
the segment and batch sizes of the reduction, bins on both sides of its two
forms."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


@pytest.mark.parametrize("scale", [1.0, 1e-160, 1e-290, 1e140, 3e-309])
@pytest.mark.parametrize("m,nbins", [(5, 1), (151, 7), (1217, 100), (19457, 128), (40_000, 129)])
def test_quotients(sg, scale, m, nbins):
    import torch
    rng = np.random.default_rng(m + nbins)
    n = 997
    score = rng.normal(size=m) * scale
    score[:: 7] = 0.0
    st = rng.choice(np.array([0, 0, 0, 1, 3], dtype=np.int8), size=m)
    n1 = rng.integers(-1, n + 2, size=m).astype(np.int32)
    got = sg.selscan_normalize(*(torch.from_numpy(a).cuda() for a in (score, st, n1)), n, nbins)
    g = {k: v.cpu().numpy() for k, v in got.items() if not k.startswith("_")}
    b = np.clip(n1.astype(np.int64) * nbins // n, 0, nbins - 1)
    b[n1 <= 0] = 0
    with np.errstate(all="ignore"):
        want = (score - g["mean"][b]) / g["sd"][b]
    ok = (st == 0) & (g["count"][b] >= 2) & (g["sd"][b] > 0)
    assert np.array_equal(np.isnan(g["score"]), ~ok | np.isnan(want))
    assert np.array_equal(g["score"][ok], want[ok], equal_nan=True)
    if scale == 1.0:
        ref = oracle.normalize(score, st, np.clip(n1, 0, n).astype(np.int32), n, nbins)
        assert np.array_equal(g["count"], ref["count"])
        np.testing.assert_allclose(g["sd"][ref["count"] > 1], ref["sd"][ref["count"] > 1], rtol=1e-12)
