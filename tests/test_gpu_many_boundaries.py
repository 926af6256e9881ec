"""Walks whose first 32 steps have more run boundaries than the on-chip list holds
(1,024; unlinked or very large samples): the sorted forms take windows of fewer
steps, and where one window still does not fit, its list runs on in global
memory.  Every bit of the per-step walk: walks of a dozen steps beside walks to
the end of a long identical stretch, one class of each, samples around the
list's size and at the sweep's limit."""
import numpy as np
import pytest

import synth
from parity_util import assert_bitwise_equal
from test_gpu_chunk_scan import scan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def unlinked(n, m, seed, same=0):
    """Independent alleles, the first `same` haplotypes alike over the middle."""
    rng = np.random.default_rng(seed)
    hap = (rng.random((m, n)) < rng.random((m, 1)) ** 2).astype(np.uint8)
    if same:
        hap[m // 4: 3 * m // 4, :same] = hap[m // 4: 3 * m // 4, :1]
        hap[m // 2, :] = 0
        hap[m // 2, :same] = 1
    pos = np.cumsum(rng.integers(1, 400, size=m)).astype(np.int64)
    return hap, pos, pos * 1e-6


@pytest.mark.parametrize("n", [1025, 1100, 1500, 2100, 4100, 6144, 9000, 16_383])
@pytest.mark.parametrize("same", [0, 3])
def test_ihs(sg, n, same):
    m = 300 if n < 5000 else 150
    hap, pos, gmap = unlinked(n, m, n + same, same * n // 5)
    rows = synth.pack(hap)
    want = scan(sg, rows, pos, gmap, n, 0, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8))
    assert np.median(want["stop"][want["status"] != 1]) < 32
    for launch in (sg.make_launch(sg.SCHED_IN_ORDER), sg.make_launch(sg.SCHED_SWEEP),
                   sg.make_launch(sg.SCHED_SWEEP, sweep_warmup=16, sweep_stage_cores=40)):
        assert_bitwise_equal(want, scan(sg, rows, pos, gmap, n, 0, launch))


@pytest.mark.parametrize("nA,nB", [(700, 600), (2500, 1700), (6000, 7000)])
def test_xpehh(sg, nA, nB):
    hap, pos, gmap = unlinked(nA + nB, 150, nA, nA // 2)
    rows = np.concatenate([synth.pack(hap[:, :nA]), synth.pack(hap[:, nA:])], 1)
    want = scan(sg, rows, pos, gmap, nA, nB, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8))
    for launch in (sg.make_launch(sg.SCHED_IN_ORDER), sg.make_launch(sg.SCHED_SWEEP)):
        assert_bitwise_equal(want, scan(sg, rows, pos, gmap, nA, nB, launch))


def test_core_range(sg):
    """Slots that a walking warp puts by, in a range that starts inside the chromosome."""
    from parity_util import to_np
    n, m, k0, k1 = 4100, 300, 37, 251
    hap, pos, gmap = unlinked(n, m, 9, n // 2)
    rows = synth.pack(hap)
    want = scan(sg, rows, pos, gmap, n, 0, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8))
    h, p, g = sg.to_device(rows, pos, gmap)
    for kw in (dict(), dict(sweep_stage_cores=17)):
        out = sg.selscan_ihs_range(h, n, p, g, k0, k1, launch=sg.make_launch(sg.SCHED_SWEEP, **kw))
        sg.check(out)
        assert_bitwise_equal({f: v[k0:k1] for f, v in want.items()}, to_np(out))
