"""Standardised scores at the ends of FP64's range are the quotients (score -
mean) / SD of the statistics that are returned, as the divide gives them: 0 in a
bin whose SD overflowed, and from SDs (handed to the shard form) whose
reciprocal is subnormal, zero or infinite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def quotients(score, mean, sd, count, b):
    with np.errstate(all="ignore"):
        q = (score - mean[b]) / sd[b]
    return np.where((count[b] >= 2) & (sd[b] > 0), q, np.nan)


@pytest.mark.parametrize("scale", [1e153, 1e155, 1e200, 1e300, 1e306])
@pytest.mark.parametrize("m,nbins", [(1217, 100), (3000, 129)])
def test_overflowing_sd(sg, scale, m, nbins):
    import torch
    rng = np.random.default_rng(m)
    n, n1 = 997, rng.integers(0, 998, size=m).astype(np.int32)
    score = rng.normal(size=m) * scale
    g = sg.selscan_normalize(torch.from_numpy(score).cuda(), torch.zeros(m, dtype=torch.int8, device="cuda"),
                             torch.from_numpy(n1).cuda(), n, nbins)
    g = {k: v.cpu().numpy() for k, v in g.items() if not k.startswith("_")}
    b = np.minimum(n1.astype(np.int64) * nbins // n, nbins - 1)
    want = quotients(score, g["mean"], g["sd"], g["count"], b)
    assert np.isinf(g["sd"]).any() == (scale > 1e154) and np.isfinite(want).any()
    np.testing.assert_array_equal(g["score"], want)


@pytest.mark.parametrize("sd", [5e-324, 1e-310, 5e-309, 1e-308, 1.1e-300, 1.0, 1e300, 6.7e307, 1.7e308, np.inf])
@pytest.mark.parametrize("scale", [3e-308, 1e-250, 1.0, 1e250, 1e308])
def test_any_sd(sg, sd, scale):
    import torch
    rng = np.random.default_rng(7)
    m = 4099
    score = rng.uniform(-1.0, 1.0, size=m) * scale
    score[:4] = [np.inf, -np.inf, np.nan, 0.0]
    stat = np.array([0.0]), np.array([sd]), np.array([m])
    got = sg.selscan_normalize_apply(torch.from_numpy(score).cuda(), torch.zeros(m, dtype=torch.int8, device="cuda"),
                                     torch.zeros(m, dtype=torch.int32, device="cuda"), 10, 1,
                                     *(torch.from_numpy(stat[i]).cuda() for i in (2, 0, 1))).cpu().numpy()
    np.testing.assert_array_equal(got, quotients(score, stat[0], stat[1], stat[2], np.zeros(m, np.int64)))
