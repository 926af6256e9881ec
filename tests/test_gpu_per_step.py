"""The per-step walk against the oracle under every rule and parameter, beside
the sorted forms: it still runs core ranges, samples above 6,144 haplotypes below
the sweep's line, small workspaces and second passes, and a default launch of a
short chromosome no longer reaches it."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import assert_ihs_equal, assert_xpehh_equal, to_np

pytestmark = pytest.mark.gpu

FORMS = dict(per_step=dict(schedule=1, warps_per_cta=8), longest_first=dict(schedule=0, probe_steps=2),
             plain=dict(schedule=2), one_launch=dict(schedule=1), sweep=dict(schedule=3))


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1403_6854_gb300 as sg
    return sg


def run(sg, rows, nA, nB, pos, gmap, form, k=None, **params):
    h, p, g = sg.to_device(rows, pos, gmap)
    kw = dict(params=sg.selscan_default_params(**params), launch=sg.make_launch(**FORMS[form]) if form else None)
    k = k or (0, rows.shape[0])
    out = (sg.selscan_xpehh_range(h, nA, nB, p, g, *k, **kw) if nB else sg.selscan_ihs_range(h, nA, p, g, *k, **kw))
    sg.check(out)
    return to_np(out)


def compare(sg, rows, nA, nB, pos, gmap, form, k=None, clean=None, **params):
    got = run(sg, rows, nA, nB, pos, gmap, form, k, **params)
    clean = rows if clean is None else clean
    op = oracle.params(**params)
    ref = oracle.xpehh(clean, nA, nB, pos, gmap, p=op) if nB else oracle.ihs(clean, nA, pos, gmap, p=op)
    if k is not None:
        ref = {f: v[k[0]:k[1]] for f, v in ref.items()}
    (assert_xpehh_equal if nB else assert_ihs_equal)(got, ref)


def gapped(n, m, seed):
    hap, pos, gmap = synth.tiny_mosaic(n, m, seed, founders=3, switch=0.03, flip=0.01, dyadic_map=False)
    steps = np.diff(pos)
    steps[np.linspace(5, m - 10, 6).astype(int)] = [20_000, 20_001, 200_000, 200_001, 45_000, 1_000_000]
    return hap, np.concatenate([pos[:1], pos[0] + np.cumsum(steps)]).astype(np.int64), gmap


def packed(hap, nA, pad=0):
    """Rows of A's words then B's, and a copy whose pad bits and words are set."""
    parts = [hap[:, :nA]] + ([hap[:, nA:]] if hap.shape[1] > nA else [])
    clean = np.concatenate([synth.pack(p) for p in parts] + [np.zeros((hap.shape[0], pad), np.uint64)], 1)
    dirty, w = clean.copy(), 0
    for p in parts:
        n, w = p.shape[1], w + (p.shape[1] + 63) // 64
        if n % 64:
            dirty[:, w - 1] |= np.uint64(0xFFFFFFFFFFFFFFFF) << np.uint64(n % 64)
    dirty[:, w:] = np.uint64(0xDEADBEEFDEADBEEF)
    return clean, dirty


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("nB", [0, 23])
@pytest.mark.parametrize("params", [dict(), dict(include_crossing_term=1), dict(ehh_cut=(1, 4)),
                                    dict(ehh_cut=(3, 100)), dict(gap_scale_bp=5000, max_gap_bp=60_000),
                                    dict(maf=(1, 5), xpehh_maf_filter=1), dict(use_physical_map=1),
                                    dict(use_physical_map=1, include_crossing_term=1)])
def test_rules_and_parameters(sg, form, nB, params):
    """Gaps at and around both limits, dirty pad bits and words, every parameter;
    the physical map beside a decreasing genetic one, which must not be read."""
    nA = 70 if nB == 0 else 47
    hap, pos, gmap = gapped(nA + nB, 90, 11 + nB)
    clean, dirty = packed(hap, nA, pad=2)
    gmap = gmap[::-1].copy() if params.get("use_physical_map") else gmap
    compare(sg, dirty, nA, nB, pos, gmap, form, clean=clean, **params)


@pytest.mark.parametrize("nB", [0, 65])
@pytest.mark.parametrize("k", [(0, 1), (17, 150), (299, 300), (0, 299), (1, 300)])
@pytest.mark.parametrize("params", [dict(), dict(use_physical_map=1, include_crossing_term=1)])
def test_core_ranges(sg, nB, k, params):
    hap, pos, gmap = gapped(130 + nB, 300, 5)
    clean, dirty = packed(hap, 130, pad=1)
    compare(sg, dirty, 130, nB, pos, gmap, None, k, clean=clean, **params)


@pytest.mark.parametrize("nA,nB", [(6145, 0), (3073, 3073)])
def test_large_samples_of_short_chromosomes(sg, nA, nB):
    hap, pos, gmap = gapped(nA + nB, 40, 3)
    clean, dirty = packed(hap, nA)
    compare(sg, dirty, nA, nB, pos, gmap, None, clean=clean)
