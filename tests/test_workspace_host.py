"""Workspace sizes that need no GPU: what a default call asks for against the
forms that it can also run in."""
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
