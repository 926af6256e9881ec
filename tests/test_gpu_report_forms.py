"""A single-locus report runs its walks step by step beside the sorted form and
takes whichever is done first: walks of a few steps, of some hundred (some of the
six long, some short), to the array's end and past the sorted form's 2,048 steps,
with sample sizes on both sides of each CTA width, equal the per-step form's bits
(a workspace without room for the sorted form) again and again."""
import numpy as np
import pytest

import synth
from parity_util import assert_bitwise_equal, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


@pytest.mark.parametrize("n", [2, 33, 204, 512, 513, 2048, 2049, 5000, 10_500])
@pytest.mark.parametrize("switch", [0.4, 0.02, 0.0])
def test_either_form_same_bits(sg, n, switch):
    import torch
    m = 5200 if n <= 512 else 700
    hap, pos, gmap = synth.tiny_mosaic(n, m, n, founders=3, switch=switch, flip=0.0 if switch == 0.0 else 0.002)
    hap[m // 2 + 3:, : n // 2] = hap[m // 2 + 3:, :1]             # long in one direction and class
    h, p, g = sg.to_device(synth.pack(hap), pos, gmap)
    raw = torch.empty(sg.selscan_workspace_bytes(n, m, sg.MODE_EHH) + 256, dtype=torch.uint8, device="cuda")
    ws = raw[(-raw.data_ptr()) % 256:]
    for locus in (0, 40, m // 2, m - 1):
        step = sg.selscan_ehh(h, n, p, g, locus, 64, workspace=ws[:sg.selscan_workspace_min_bytes(n, m, sg.MODE_EHH)])
        sg.check(step)
        want = to_np(step)
        for _ in range(5):
            out = sg.selscan_ehh(h, n, p, g, locus, 64, workspace=ws)
            sg.check(out)
            assert_bitwise_equal(want, to_np(out))
