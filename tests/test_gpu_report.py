"""The single-locus report from the sorted state, bit for bit with the report of
the per-step walks (selscan_ehh_noalloc) and against the oracle: samples at the
changes of CTA width, loci at the array's ends and next to 32-marker words,
walks that outlive the 2,048 markers of history on either side (left to the
per-step walk one by one), gaps, one-allele loci, truncated traces."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


@pytest.mark.parametrize("n,m", [(2, 40), (100, 9000), (513, 5000), (1025, 2300), (2100, 700), (6145, 300)])
@pytest.mark.parametrize("kind", ["mosaic", "long"])
def test_equals_per_step_report(sg, n, m, kind):
    hap, pos, gmap = synth.tiny_mosaic(n, m, n + m, founders=6, switch=0.02 if kind == "mosaic" else 0.0005,
                                       flip=0.003 if kind == "mosaic" else 0.0)
    if kind == "long":
        hap[:, n // 2:] = hap[:, :1]                      # half the sample identical everywhere
        hap[m // 2] = 0
        hap[m // 2, n // 2:] = 1
    else:
        pos[2 * m // 3:] += 30_000
        pos[3 * m // 4:] += 300_000
        hap[m // 3] = 1                                    # a locus without allele 0
    rows = synth.pack(hap, ld=(n + 63) // 64 + 1)
    h, p, g = sg.to_device(rows, pos, gmap)
    for locus in sorted({0, 1, 31 % m, 32 % m, m // 3, m // 2, m - 2, m - 1}):
        for cap in (0, 3, 4096):
            a = sg.selscan_ehh(h, n, p, g, locus, cap)
            sg.check(a)
            a = to_np(a)
            b = to_np(sg.selscan_ehh_noalloc(h, n, p, g, locus, cap))
            for f in a:
                assert np.array_equal(a[f], b[f]), (f, locus, cap)
    locus = m // 2
    ref = oracle.ehh(rows, n, pos, gmap, locus, 4096)
    assert np.array_equal(a["len"].shape, ref["len"].shape)
    a = to_np(sg.selscan_ehh(h, n, p, g, locus, 4096))
    for f in ("len", "stop", "status", "denom"):
        assert np.array_equal(a[f], ref[f]), f
    np.testing.assert_allclose(a["ihh"], ref["ihh"], rtol=1e-12, atol=0)


def test_smaller_workspaces_same_bits(sg):
    """Down to the first workspace that is refused; those without room for the
    sorted form take the per-step walks."""
    import torch
    n, m, locus = 300, 900, 450
    hap, pos, gmap = synth.tiny_mosaic(n, m, 5, founders=6, switch=0.02, flip=0.003)
    h, p, g = sg.to_device(synth.pack(hap), pos, gmap)
    full = sg.selscan_workspace_bytes(n, m, sg.MODE_EHH)
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:][:full]
    lib, first = sg.load_library(), None
    for pct in range(100, 0, -1):
        out = dict(S=torch.zeros((3, 2, 64), dtype=torch.int64, device="cuda"),
                   **{f: torch.empty((3, 2), dtype=d, device="cuda") for f, d in
                      (("len", torch.int64), ("stop", torch.int32), ("status", torch.int8), ("ihh", torch.float64))},
                   denom=torch.empty(3, dtype=torch.int64, device="cuda"),
                   error=torch.zeros(1, dtype=torch.int32, device="cuda"))
        o = sg.selscan_ehh_out(*(out[f].data_ptr() for f in ("S", "len", "stop", "status", "ihh", "denom", "error")))
        rc = lib.selscan_ehh(h.data_ptr(), h.shape[1], n, m, p.data_ptr(), g.data_ptr(), locus,
                             sg.selscan_default_params(), o, 64, ws.data_ptr(), full * pct // 100, None)
        if rc == sg.ERR_WORKSPACE:
            break
        assert rc == sg.OK
        torch.cuda.synchronize()
        sg.check(out)
        first = first or to_np(out)
        for f, v in to_np(out).items():
            assert np.array_equal(first[f], v), f
    assert 1 < pct < 99
