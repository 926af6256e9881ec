"""Scans and reports through the binding in a workspace sized for a larger
sample, where it has no room for the starting states' words or the report's
sorted form: the same bits as in a workspace of their own."""
import numpy as np
import pytest

from parity_util import assert_bitwise_equal, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def inputs(sg, n, m):
    rng = np.random.default_rng(n)
    rows = rng.integers(0, 1 << 63, size=(m, (n + 63) // 64), dtype=np.uint64)
    rows[m // 3: m // 3 + 200] = rows[m // 3] & np.uint64(0x0FF0FF0FF0FF0FF0)     # long walks
    pos = np.cumsum(rng.integers(1, 400, size=m)).astype(np.int64)
    return sg.to_device(rows, pos, pos * 1e-6)


def sized_for(sg, n, m, mode, small):
    import torch
    full = sg.selscan_workspace_bytes(n, m, mode)
    assert full < sg.selscan_workspace_bytes(small, m, mode)
    raw = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    return raw[(-raw.data_ptr()) % 256:][:full]


@pytest.mark.parametrize("nA,nB", [(10_496, 0), (5248, 5248)])
def test_scan_in_a_larger_samples_workspace(sg, nA, nB):
    n, m = nA + nB, 76_000
    h, p, g = inputs(sg, n, m)
    mode = sg.MODE_XPEHH if nB else sg.MODE_IHS
    outs = []
    for ws in (None, sized_for(sg, 10_600, m, mode, n)):
        if nB:
            out = sg.selscan_xpehh(h, nA, nB, p, g, workspace=ws)
        else:
            out = sg.selscan_ihs(h, n, p, g, workspace=ws)
        sg.check(out)
        outs.append(to_np(out))
    assert_bitwise_equal(*outs)


def test_report_in_a_larger_samples_workspace(sg):
    n, m = 10_496, 900
    h, p, g = inputs(sg, n, m)
    for locus in (0, m // 3 + 50, m - 1):
        outs = []
        for ws in (None, sized_for(sg, 10_600, m, sg.MODE_EHH, n)):
            out = sg.selscan_ehh(h, n, p, g, locus, 64, workspace=ws)
            sg.check(out)
            outs.append(to_np(out))
        assert_bitwise_equal(*outs)
