"""Starting states of the sorted sweep's chunks, sorted directly from the
history's 32-marker words, against the oracle: history lengths around word
boundaries (so that the nearest and the farthest word are partial, also both
in one word), samples around the sizes at which all, or only the late, rounds
run on the listed unresolved haplotypes, rows with pad words, core ranges
(the words of a range start at its first history marker), and haplotypes that
stay identical over the whole history."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import assert_ihs_equal, assert_xpehh_equal, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def mosaic(n, m, seed):
    """Near-copies of a few founders, a third of them exact copies of one."""
    hap, pos, gmap = synth.tiny_mosaic(n, m, seed, founders=6, switch=0.03, flip=0.004)
    hap[:, : n // 3] = hap[:, :1]
    return hap, pos, gmap


@pytest.mark.parametrize("n", [2, 65, 511, 513, 1024, 1025, 2049, 2500])
@pytest.mark.parametrize("warmup", [16, 31, 33, 64, 95, 0])
def test_history_lengths(sg, n, warmup):
    m = 600
    hap, pos, gmap = mosaic(n, m, 7 * n + warmup)
    rows = synth.pack(hap, ld=(n + 63) // 64 + 1)
    cores = np.array([0, 1, 31, 32, 200, 255, 256, 257, 299, 300, 301, 350, 598, 599])
    ref = oracle.ihs(rows, n, pos, gmap, cores=cores)
    h, p, g = sg.to_device(rows, pos, gmap)
    out = sg.selscan_ihs(h, n, p, g, launch=sg.make_launch(sg.SCHED_SWEEP, sweep_warmup=warmup))
    sg.check(out)
    assert_ihs_equal(to_np(out), ref, idx=cores)


@pytest.mark.parametrize("k0,k1", [(0, 300), (299, 563), (37, 599)])
def test_range_with_two_populations(sg, k0, k1):
    nA, nB, m = 130, 95, 600
    hap, pos, gmap = mosaic(nA + nB, m, k0)
    rows = np.concatenate([synth.pack(hap[:, :nA]), synth.pack(hap[:, nA:])], 1)
    ref = oracle.xpehh(rows, nA, nB, pos, gmap)
    h, p, g = sg.to_device(rows, pos, gmap)
    out = sg.selscan_xpehh_range(h, nA, nB, p, g, k0, k1,
                                 launch=sg.make_launch(sg.SCHED_SWEEP, sweep_warmup=70))
    sg.check(out)
    assert_xpehh_equal(to_np(out), {k: v[k0:k1] for k, v in ref.items()})
