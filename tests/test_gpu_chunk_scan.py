"""Short scans in one launch (the in-order schedule without a per-step launch
field) against the oracle and, bit for bit, against the per-step walk: sample
sizes around each change of sorting width, chromosomes of one marker up to
several chunks per SM and across the change of CTA shape, walks that run to the
array ends and over the whole chromosome, gaps, and XPEHH."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import assert_bitwise_equal, assert_ihs_equal, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def scan(sg, rows, pos, gmap, nA, nB, launch):
    h, p, g = sg.to_device(rows, pos, gmap)
    out = sg.selscan_xpehh(h, nA, nB, p, g, launch=launch) if nB else sg.selscan_ihs(h, nA, p, g, launch=launch)
    sg.check(out)
    return to_np(out)


@pytest.mark.parametrize("n", [2, 100, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4000])
@pytest.mark.parametrize("m", [1, 3, 304, 700])
def test_sizes_match_oracle(sg, n, m):
    hap, pos, gmap = synth.tiny_mosaic(n, m, 31 * n + m, founders=5, switch=0.04, flip=0.01)
    hap[:, : n // 4] = hap[:, :1]
    if m > 300:
        pos[m // 2:] += 250_000                       # a gap abort in the middle
    rows = synth.pack(hap)
    cores = np.unique(np.array([0, 1, m // 3, m // 2 - 1, m // 2, m - 1]).clip(0, m - 1))
    ref = oracle.ihs(rows, n, pos, gmap, cores=cores)
    assert_ihs_equal(scan(sg, rows, pos, gmap, n, 0, sg.make_launch(sg.SCHED_IN_ORDER)), ref, idx=cores)


@pytest.mark.parametrize("nA,nB,m", [(60, 44, 4863), (60, 44, 4864), (130, 127, 4863), (130, 127, 6000),
                                     (300, 213, 5000), (700, 500, 2500), (204, 0, 9000), (1025, 0, 3000)])
def test_equals_per_step_walk(sg, nA, nB, m):
    """Every output bit of the per-step walk (a launch field of its own takes
    it), with an identical stretch over a third of the chromosome."""
    n = nA + nB
    hap, pos, gmap = synth.tiny_mosaic(n, m, n + m, founders=8, switch=0.01, flip=0.002)
    hap[m // 3: 2 * m // 3, : n // 3] = hap[m // 3: 2 * m // 3, :1]
    parts = [synth.pack(hap[:, :nA])] + ([synth.pack(hap[:, nA:])] if nB else [])
    rows = np.concatenate(parts, 1)
    a = scan(sg, rows, pos, gmap, nA, nB, sg.make_launch(sg.SCHED_IN_ORDER))
    b = scan(sg, rows, pos, gmap, nA, nB, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8))
    assert_bitwise_equal(b, a)
