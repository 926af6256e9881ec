"""Both forms of a tick: the per-step walk (a scan with more than 65,000 markers
or 6,144 haplotypes, or a workspace without room for the sorted form) and the
sorted chunks, with the bits of the scan alone; scans that have no cores in a
tick take no part in it."""
import numpy as np
import pytest

import synth
from parity_util import assert_bitwise_equal, to_np
from test_gpu_chunk_scan import batch_scan, scan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def make(sg, sizes):
    scans, alone = [], []
    for i, (nA, nB, m) in enumerate(sizes):
        hap, pos, gmap = synth.tiny_mosaic(nA + nB, m, 55 + i, founders=6, switch=0.02, flip=0.004)
        rows = np.concatenate([synth.pack(hap[:, :nA])] + ([synth.pack(hap[:, nA:])] if nB else []), 1)
        scans.append(batch_scan(sg, rows, pos, gmap, nA, nB))
        alone.append(scan(sg, rows, pos, gmap, nA, nB, sg.make_launch(sg.SCHED_IN_ORDER, warps_per_cta=8)))
    return scans, alone, max(s.nA + s.nB for s, _, _ in scans), max(s.ld for s, _, _ in scans)


def workspace(nb):
    import torch
    raw = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    return raw[(-raw.data_ptr()) % 256:][:nb]


def check(sg, scans, alone, idx):
    for i in idx:
        s, t, _ = scans[i]
        sg.selscan_batch_finalize(s)
        got, ref = to_np(t), dict(alone[i])
        assert int(t["error"].item()) == 0
        a, b = ("ihhA", "ihhB") if s.nB else ("ihh1", "ihh0")
        assert_bitwise_equal(got, {**ref, "ihh_a": ref.pop(a), "ihh_b": ref.pop(b)})


@pytest.mark.parametrize("sizes", [[(40, 0, 65_001), (30, 33, 500), (200, 0, 900)],
                                   [(6145, 0, 40), (64, 0, 700), (3100, 3100, 33)]])
def test_per_step_ticks_equal_scans_alone(sg, sizes):
    scans, alone, max_n, max_ld = make(sg, sizes)
    ws = workspace(sg.selscan_batch_workspace_bytes(max_n, max_ld, len(scans), 256))
    for s, _, _ in scans:
        sg.selscan_batch_prepare(s)
    cuts = [(i, a, b) for i, (s, _, _) in enumerate(scans) for a, b in ((0, s.m // 3), (s.m // 3, s.m))]
    sg.selscan_batch_run([s for s, _, _ in scans], *zip(*cuts), max_n, max_ld, ws)
    check(sg, scans, alone, range(len(scans)))


def test_workspaces_down_to_the_per_step_walks(sg):
    """From the size for the tick's bounds down to the first that is refused:
    those without room for the chunks take the per-step walk."""
    scans, alone, max_n, max_ld = make(sg, [(300, 0, 9000), (100, 150, 6000)])
    full = sg.selscan_batch_workspace_bytes(max_n, max_ld, len(scans), 256)
    ws, served = workspace(full), 0
    for pct in range(100, 0, -3):
        for s, _, _ in scans:
            sg.selscan_batch_prepare(s)
        try:
            sg.selscan_batch_run([s for s, _, _ in scans], [0, 1], [0, 0], [s.m for s, _, _ in scans], max_n, max_ld,
                                 ws[:full * pct // 100])
        except sg.SelscanError as e:
            assert e.code == sg.ERR_WORKSPACE
            break
        served += 1
        check(sg, scans, alone, range(2))
    assert 1 < served < 33


def test_scans_without_cores_take_no_part(sg):
    """A resident scan without cores in the tick costs it nothing: neither its
    words nor, above the sorted form's limits, the other scans' form."""
    import torch
    scans, alone, max_n, max_ld = make(sg, [(100, 0, 600), (2000, 0, 9000), (7000, 0, 40), (30, 0, 65_100)])
    nb = sg.selscan_batch_workspace_bytes(max_n, max_ld, len(scans), 256)
    ws = workspace(nb)
    ws.zero_()
    for s, _, _ in scans:
        sg.selscan_batch_prepare(s)
    before = [{f: t.clone() for f, t in ts.items()} for _, ts, _ in scans]
    sg.selscan_batch_run([s for s, _, _ in scans], [0, 1, 3], [0, 50, 7], [scans[0][0].m, 50, 7], max_n, max_ld, ws)
    torch.cuda.synchronize()
    # the words, states, slots and flags of 100 haplotypes x 600 markers; the words of 2,000 x 9,000 are 2.3 MB
    assert 100_000 < int(torch.count_nonzero(ws.view(torch.int64))) * 8 < 1_000_000
    for (_, ts, _), b in zip(scans[1:], before[1:]):
        for f, t in ts.items():
            assert torch.equal(t.view(torch.uint8), b[f].view(torch.uint8)), f
    check(sg, scans, alone, [0])
