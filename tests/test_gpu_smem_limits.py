"""Scans of two host threads, each with its own stream and workspace, while a
third asks for sizes: no call changes what another's launch may use."""
import threading

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


@pytest.mark.parametrize("big,small,schedule", [(5000, 2100, 1), (2000, 1100, 1), (5000, 4100, 3), (4000, 2400, 0)])
def test_threads_of_different_samples(sg, big, small, schedule):
    import torch
    m, failed, stop = 40, [], threading.Event()
    launch = sg.make_launch(schedule)

    def work(n, reps):
        try:
            hap, pos, gmap = synth.tiny_mosaic(n, m, n, founders=6, switch=0.02, flip=0.004)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                h, p, g = sg.to_device(synth.pack(hap), pos, gmap)
                ws = torch.empty(sg.selscan_workspace_bytes(n, m, sg.MODE_IHS, launch) + 256, dtype=torch.uint8,
                                 device="cuda")
                ws = ws[(-ws.data_ptr()) % 256:]
                first = None
                for _ in range(reps):
                    out = sg.selscan_ihs(h, n, p, g, launch=launch, workspace=ws, stream=s)
                    sg.selscan_ehh(h, n, p, g, m // 2, 16, stream=s)
                    s.synchronize()
                    sg.check(out)
                    first = first or to_np(out)
                    assert_bitwise_equal(first, to_np(out))
        except Exception as e:                    # reported by the main thread
            failed.append(e)

    def ask():
        while not stop.is_set():
            for n in (small, 100, big):
                sg.selscan_workspace_bytes(n, m, sg.MODE_IHS, launch)

    work(big, 1)                                  # modules loaded before the threads meet
    work(small, 1)
    asker = threading.Thread(target=ask)
    asker.start()
    ts = [threading.Thread(target=work, args=(n, 150)) for n in (big, small)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    stop.set()
    asker.join()
    assert not failed, failed[0]
