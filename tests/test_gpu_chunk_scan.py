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


def batch_scan(sg, rows, pos, gmap, nA, nB):
    import torch
    hap, p, g = sg.to_device(rows, pos, gmap)
    m, mode = hap.shape[0], sg.MODE_XPEHH if nB else sg.MODE_IHS
    ipc, nd = (2, 6) if nB else (4, 4)
    e = lambda shape, dt: torch.empty(shape, dtype=dt, device="cuda")
    t = dict(status=e(m, torch.int8), n1=e(m, torch.int32), ihh_a=e(m, torch.float64), ihh_b=e(m, torch.float64),
             lnratio=e(m, torch.float64), stop=e((m, ipc), torch.int32), digest=e((m, nd), torch.int64),
             error=torch.zeros(1, dtype=torch.int32, device="cuda"))
    raw = e(sg.selscan_batch_item_bytes(m, mode) + 256, torch.uint8)
    s = sg.selscan_scan()
    s.mode, s.nA, s.nB, s.m, s.ld, s.params = mode, nA, nB, m, hap.shape[1], sg.selscan_default_params()
    s.hap, s.pos_bp, s.gmap = hap.data_ptr(), p.data_ptr(), g.data_ptr()
    s.items = raw.data_ptr() + (-raw.data_ptr()) % 256
    for f, v in t.items():
        setattr(s, f, v.data_ptr())
    return s, t, (hap, p, g, raw)


@pytest.mark.parametrize("sizes", [[(30, 0, 900), (200, 250, 1300), (512, 0, 700)],
                                   [(1000, 0, 800), (40, 33, 2100), (2, 0, 5)],
                                   [(100, 0, 1500), (900, 800, 600), (1500, 0, 333), (64, 0, 64)],
                                   [(2300, 0, 400), (77, 0, 1000), (1200, 1300, 350)]])
def test_ticks_equal_scans_alone(sg, sizes):
    """Two ticks over uneven core ranges of scans of different samples and both
    kinds (empty ranges among them): every output bit of the scan alone."""
    import torch
    scans, alone = [], []
    for i, (nA, nB, m) in enumerate(sizes):
        hap, pos, gmap = synth.tiny_mosaic(nA + nB, m, 77 + i, founders=6, switch=0.02, flip=0.004)
        parts = [synth.pack(hap[:, :nA])] + ([synth.pack(hap[:, nA:])] if nB else [])
        rows = np.concatenate(parts, 1)
        scans.append(batch_scan(sg, rows, pos, gmap, nA, nB))
        alone.append(scan(sg, rows, pos, gmap, nA, nB, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8)))
    max_n, max_ld = max(s.nA + s.nB for s, _, _ in scans), max(s.ld for s, _, _ in scans)
    nb = sg.selscan_batch_workspace_bytes(max_n, max_ld, len(scans), 256)
    raw = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    off = (-raw.data_ptr()) % 256
    units = [[], []]
    for i, (s, _, _) in enumerate(scans):
        sg.selscan_batch_prepare(s)
        cuts = sorted({0, s.m // 7, s.m // 3, s.m // 3 + 1, s.m})
        for q, (a, b) in enumerate(zip(cuts, cuts[1:])):
            units[q % 2].append((i, a, b))
        units[i % 2].append((i, s.m // 2, s.m // 2))
    for us in units:
        sg.selscan_batch_run([s for s, _, _ in scans], *zip(*us), max_n, max_ld, raw[off:off + nb])
    for (s, t, _), ref in zip(scans, alone):
        sg.selscan_batch_finalize(s)
        got = to_np(t)
        assert int(t["error"].item()) == 0
        a, b = ("ihhA", "ihhB") if s.nB else ("ihh1", "ihh0")
        ref = {**ref, "ihh_a": ref.pop(a), "ihh_b": ref.pop(b)}
        assert_bitwise_equal(got, ref)


@pytest.mark.parametrize("n,m", [(513, 2400), (600, 40_000)])
def test_smaller_workspaces_same_bits(sg, n, m):
    """Workspaces one percent smaller each time, down to the first that is
    refused: those without room for the chunks' slots (in-order) or for the
    starting states' words (sweep) take the per-step walk or swept histories,
    with the same bits."""
    import torch
    hap, pos, gmap = synth.tiny_mosaic(n, m, n + m, founders=8, switch=0.02, flip=0.002)
    h, p, g = sg.to_device(synth.pack(hap), pos, gmap)
    full = sg.selscan_workspace_bytes(n, m, sg.MODE_IHS)
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:][:full]
    lib, first = sg.load_library(), None
    for pct in range(100, 0, -1):
        out = sg._ihs_outputs(m, h.device)
        o = sg.selscan_ihs_out(*(out[f].data_ptr() for f in ("status", "n1", "ihh1", "ihh0", "lnratio",
                                                             "stop", "digest", "error")))
        rc = lib.selscan_ihs(h.data_ptr(), h.shape[1], n, m, p.data_ptr(), g.data_ptr(),
                             sg.selscan_default_params(), o, ws.data_ptr(), full * pct // 100, None, None)
        if rc == sg.ERR_WORKSPACE:
            break
        assert rc == sg.OK
        torch.cuda.synchronize()
        sg.check(out)
        first = first or to_np(out)
        assert_bitwise_equal(first, to_np(out))
    assert 1 < pct < 99
