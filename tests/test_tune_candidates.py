"""The autotuner always times what a default launch would do: otherwise it could
hand out a slower shape than no shape at all."""
import pytest

from paper_1403_6854_gb300.tune import DEFAULT_CANDIDATES, SWEEP_CANDIDATES, SWEEP_MAX_N


@pytest.mark.parametrize("n,m", [(100, 2000), (204, 22147), (2000, 12_724), (5000, 52_000), (1000, 200_000),
                                 (5000, 1_000_000), (16_383, 90_000)])
def test_default_form_is_a_candidate(n, m):
    from paper_1403_6854_gb300 import _build
    _build.build()
    import paper_1403_6854_gb300 as sg
    for mode in (sg.MODE_IHS, sg.MODE_XPEHH):
        assert n <= SWEEP_MAX_N and dict(schedule=sg.selscan_default_schedule(n, m, mode)) in SWEEP_CANDIDATES


def test_per_step_candidates_hold_the_default():
    """Above the sweep's sample limit a default launch walks every step with 8
    warps per CTA and 512 group words."""
    assert dict(schedule=1, warps_per_cta=8, smem_entries=512, window_rows=0, cores_per_fetch=1) in DEFAULT_CANDIDATES
