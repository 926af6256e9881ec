"""Workspace sizes that need no GPU: what a default call asks for against the
forms that it can also run in."""
import itertools

import pytest


@pytest.fixture(scope="module")
def sg():
    from paper_1403_6854_gb300 import _build
    _build.build()
    import paper_1403_6854_gb300 as sg
    return sg


@pytest.mark.parametrize("mode", ["MODE_IHS", "MODE_XPEHH"])
@pytest.mark.parametrize("n,m", [(100, 2000), (204, 22147), (414, 22147), (1000, 36_000), (2000, 12724),
                                 (5000, 52_000), (6144, 57_000), (6000, 500), (2, 30_000)])
def test_short_scans_take_the_room_of_the_per_step_walk(sg, mode, n, m):
    """A short scan walks in one form or the other, never both: its workspace is
    that of the larger (about a fifth above the per-step walk's at the most)."""
    mode = getattr(sg, mode)
    step = sg.selscan_workspace_bytes(n, m, mode, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8))
    assert step <= sg.selscan_workspace_bytes(n, m, mode) <= 1.25 * step


@pytest.mark.parametrize("mode", ["MODE_IHS", "MODE_XPEHH", "MODE_EHH"])
def test_a_larger_shapes_workspace_serves_the_smaller(sg, mode):
    """A program that sizes its workspace once, for its largest sample and
    chromosome, passes it for the smaller ones of the same schedule too: across
    every change of form inside one (about 10,500 and 6,144 haplotypes, 65,000
    markers)."""
    mode = getattr(sg, mode)
    ns = [2, 100, 512, 513, 2000, 5000, 6144, 6145, 9000, 10_000, 10_500, 10_700, 12_000, 16_383, 16_384, 18_000]
    ms = [1, 300, 5000, 33_000, 52_000, 65_000, 65_001, 80_000, 98_000, 300_000, 1_000_000]
    full = {s: sg.selscan_workspace_bytes(*s, mode) for s in itertools.product(ns, ms)}
    sched = {s: sg.selscan_default_schedule(*s, mode) for s in full}
    least = {s: sg.selscan_workspace_min_bytes(*s, mode) for s in full}
    for n, m in full:
        assert 0 < least[n, m] <= full[n, m]
    refused = [(b, s) for b in full for s in full
               if s[0] <= b[0] and s[1] <= b[1] and sched[s] == sched[b] and least[s] > full[b]]
    assert not refused, (len(refused), refused[:5])


def test_a_passed_workspace_is_refused_below_the_least(sg):
    """The binding takes a workspace of the least size and refuses one byte less."""
    import torch
    for mode, n, m in ((sg.MODE_IHS, 10_000, 1_000_000), (sg.MODE_XPEHH, 414, 22_147), (sg.MODE_EHH, 10_400, 300)):
        least = sg.selscan_workspace_min_bytes(n, m, mode)

        class Ws:
            def __init__(self, nb): self.nb = nb
            def numel(self): return self.nb
            def element_size(self): return 1
            def data_ptr(self): return 256
        assert sg._scan_workspace(n, m, mode, None, torch.device("cuda"), Ws(least)).nb == least
        with pytest.raises(sg.SelscanError):
            sg._scan_workspace(n, m, mode, None, torch.device("cuda"), Ws(least - 1))
