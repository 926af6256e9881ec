"""Packing of unpacked bytes whose rows start anywhere: sample sizes and marker
counts around the 16-byte chunks, the 512-marker tiles, the 512-haplotype steps
and the sizes at which a row takes 8, 16 or 32 lanes; inputs that start inside a
16-byte chunk; any byte values; padded row strides."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


@pytest.mark.parametrize("n", [1, 16, 63, 113, 114, 128, 241, 242, 511, 513, 2049])
@pytest.mark.parametrize("m", [1, 15, 496, 511, 513, 1025])
@pytest.mark.parametrize("shift", [0, 1, 15])
def test_rows_anywhere(sg, n, m, shift):
    import torch
    rng = np.random.default_rng(n * 7919 + m * 31 + shift)
    h = rng.integers(0, 256, size=(m, n), dtype=np.uint8)
    for hap_major in (False, True):
        a = np.ascontiguousarray(h.T) if hap_major else h
        raw = torch.full((a.size + 32,), 255, dtype=torch.uint8, device="cuda")
        raw[shift:shift + a.size] = torch.from_numpy(a.ravel()).cuda()
        t = raw[shift:shift + a.size].view(a.shape)
        for ld in ((n + 63) // 64, (n + 63) // 64 + 33):
            got = sg.selscan_pack(t, n, hap_major=hap_major, ld=ld).cpu().numpy().view(np.uint64)
            assert np.array_equal(got, synth.pack(h, ld=ld)), (hap_major, ld)
