"""Cases whose time is this repository's performance: the scans, reports and
conversions a user of the package runs, each through its public entry points.

The inputs are Li-Stephens mosaics (founder haplotypes with a 1/k derived
allele spectrum, copied with switches along the genetic map and rare allele
errors, with planted sweeps where the case has them): the recipe of the test
and bench workloads, drawn here on the GPU from the seed alone.
"""
import numpy as np
import torch

import paper_1403_6854_gb300 as sg
from paper_1403_6854_gb300 import stream as sg_stream

SWITCH_PER_CM = 5.0
FLIP = 1e-3
GAP_AT = (0.05, 0.15, 0.30, 0.45, 0.60, 0.70, 0.80, 0.90)
GAP_BP = (20_000, 20_001, 45_000, 120_000, 200_000, 200_001, 350_000, 3_000_000)


def listed():
    return [
        # EHH decay around one locus of a chromosome-22-sized sample: the interactive report
        # behind one plot, one call at a time.
        dict(name="ehh_locus", kind="ehh", nA=204, nB=0, m=22147, founders=30, bp_per_marker=1580.0,
             sweeps=1, gaps=False, rate=1.2, spread=0.5, capacity=4096),
        # iHS on a candidate region: the smallest scan of the test configurations.
        dict(name="ihs_region", kind="ihs", nA=100, nB=0, m=2000, founders=10, bp_per_marker=1000.0,
             sweeps=0, gaps=False, rate=1.0, spread=0.0),
        # iHS on an array-typed chromosome 22 of one population, with assembly gaps.
        dict(name="ihs_chr22", kind="ihs", nA=204, nB=0, m=22147, founders=30, bp_per_marker=1580.0,
             sweeps=1, gaps=True, rate=1.2, spread=0.5),
        # XPEHH of two populations on the same chromosome.
        dict(name="xpehh_chr22", kind="xpehh", nA=204, nB=210, m=22147, founders=30,
             bp_per_marker=1580.0, sweeps=1, gaps=True, rate=1.2, spread=0.5),
        # The largest sample of the runtime tables: 2,000 haplotypes on a 4 Mb region.
        dict(name="ihs_2000", kind="ihs", nA=2000, nB=0, m=12724, founders=100, bp_per_marker=314.0,
             sweeps=0, gaps=False, rate=1.0, spread=0.0),
        # A sequenced chromosome of 1,000 haplotypes: the ordinary whole-chromosome scan.
        dict(name="ihs_200k", kind="ihs", nA=1000, nB=0, m=200_000, founders=200, bp_per_marker=250.0,
             sweeps=4, gaps=False, rate=1.2, spread=0.5),
        # The largest scans: biobank-sized panels on the longest chromosome.
        dict(name="ihs_1m", kind="ihs", nA=5000, nB=0, m=1_000_000, founders=200, bp_per_marker=250.0,
             sweeps=20, gaps=False, rate=1.2, spread=0.5),
        dict(name="xpehh_1m", kind="xpehh", nA=2500, nB=2500, m=1_000_000, founders=200,
             bp_per_marker=250.0, sweeps=20, gaps=False, rate=1.2, spread=0.5),
        # Several chromosomes in host memory scanned one after another, copies overlapped.
        dict(name="stream_3x100k", kind="stream", nA=2000, nB=0, m=100_000, founders=80,
             bp_per_marker=250.0, sweeps=2, gaps=False, rate=1.0, spread=0.0, sets=3),
        # One serving tick: short requests of mixed sizes and both statistics side by side.
        dict(name="served_tick", kind="tick", nA=100, nB=1000, m=10_000, founders=20,
             bp_per_marker=250.0, sweeps=0, gaps=False, rate=1.0, spread=0.0, scans=6),
        # Standardising a chromosome's scores in 100 frequency bins.
        dict(name="normalize_1m", kind="normalize", nA=5000, nB=0, m=1_000_000, bins=100),
        # Packing unpacked 0/1 bytes, haplotype by haplotype as phasing programs write them.
        dict(name="pack_1m", kind="pack", nA=5000, nB=0, m=1_000_000, hap_major=True),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["ihs", "ihs", "ihs", "xpehh", "xpehh", "ehh", "stream", "tick", "normalize",
                       "pack"])
    if kind == "normalize":
        return dict(kind=kind, nA=_log(rng, 50, 10_000), nB=0, m=_log(rng, 5_000, 1_000_000),
                    bins=rng.choice([1, 20, 50, 100, 100, 128]))
    if kind == "pack":
        return dict(kind=kind, nA=_log(rng, 50, 5000), nB=0, m=_log(rng, 5_000, 500_000),
                    hap_major=rng.random() < 0.6)
    n = _log(rng, 60, 6000)
    c = dict(kind=kind, nA=n, nB=0, founders=min(200, max(10, n // 25)), sweeps=rng.choice([0, 1, 3]),
             gaps=False, rate=rng.choice([1.0, 1.2]), spread=rng.choice([0.0, 0.5]),
             bp_per_marker=rng.choice([250.0, 400.0, 1000.0, 1580.0]))
    if kind == "tick":
        c.update(nA=_log(rng, 60, 300), nB=_log(rng, 400, 2000), m=_log(rng, 4_000, 20_000), founders=20,
                 scans=rng.randint(2, 10), sweeps=0, bp_per_marker=250.0)
        return c
    if kind == "stream":
        c.update(m=_log(rng, 10_000, 150_000), sets=rng.randint(2, 4))
        return c
    c["m"] = _log(rng, 2_000, 400_000 if n > 1000 else 800_000)
    c["gaps"] = c["bp_per_marker"] > 1000.0 and c["m"] > 4_000
    if kind == "ehh":
        c.update(m=min(c["m"], 200_000), capacity=rng.choice([256, 4096]))
        return c
    if kind == "xpehh":
        c.update(nA=max(40, n // 2), nB=max(41, n // 2 - rng.randint(0, n // 8)))
    # the options that are used in earnest
    opt = rng.choice(["", "", "", "crossing", "physical", "cut10"])
    if opt:
        c["option"] = opt
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream * 7919 + 17) % (1 << 62))
    return g


def _positions(case, seed):
    """int64 positions and a float64 map (cM), made on the host so that they
    are the same wherever this runs."""
    m = case["m"]
    rng = np.random.Generator(np.random.PCG64([int(seed) & 0xFFFFFFFF, m]))
    step = 1 + np.floor(rng.exponential(case["bp_per_marker"] - 1.0, m)).astype(np.int64)
    if case.get("gaps"):
        for f, b in zip(GAP_AT, GAP_BP):
            step[int(f * m)] = b
    pos = np.cumsum(step)
    seg = case["rate"] * (1.0 + case["spread"] * (2.0 * rng.random(int(pos[-1] // 1_000_000) + 2) - 1.0))
    gmap = np.cumsum(step * 1e-6 * seg[pos // 1_000_000])
    return torch.from_numpy(pos).cuda(), torch.from_numpy(gmap).cuda()


def _rows(case, seed, pos, gmap, n, founders, sweeps, stream):
    """Packed rows [m, W] of n haplotypes."""
    m, dev = pos.numel(), pos.device
    g = _gen(seed, stream)
    W = (n + 63) // 64
    dg = torch.diff(gmap, prepend=gmap[:1])
    p_switch = (1.0 - torch.exp(-SWITCH_PER_CM * dg)).float()
    w = 1.0 / torch.arange(1, founders, device=dev, dtype=torch.float64)
    rows = torch.empty((m, W), dtype=torch.int64, device=dev)
    cur = torch.randint(0, founders, (n,), generator=g, device=dev, dtype=torch.int16)
    plant = []
    for k in range(sweeps):
        u = torch.rand(2, generator=g, device=dev).tolist()
        core = int((k + 0.5) / sweeps * m)
        half = (25_000.0 + 225_000.0 * u[0]) * (case["bp_per_marker"] / 250.0) ** 0.5
        carriers = torch.rand(n, generator=g, device=dev) < 0.3 + 0.6 * u[1]
        a, b = torch.searchsorted(pos, torch.tensor([int(pos[core] - half), int(pos[core] + half)],
                                                    device=dev)).tolist()
        plant.append((a, b, core, carriers))
    step = max(16, min(m, 100_000_000 // max(n, founders) // 16 * 16))
    for k0 in range(0, m, step):
        k1 = min(m, k0 + step)
        c = k1 - k0
        count = 1 + torch.multinomial(w, c, replacement=True, generator=g)        # derived founders
        rank = torch.rand((c, founders), generator=g, device=dev).argsort(1)
        fnd = (rank < count[:, None]).to(torch.uint8)                              # [c, F]
        u = torch.rand((n, c), generator=g, device=dev)
        sw = u < p_switch[None, k0:k1]
        at = torch.where(sw, torch.arange(1, c + 1, device=dev, dtype=torch.int32), 0)
        at = torch.cummax(at, 1).values
        src = torch.randint(0, founders, (n, c + 1), generator=g, device=dev, dtype=torch.int16)
        src[:, 0] = cur
        src = src.gather(1, at.long())
        cur = src[:, -1].clone()
        del at, sw
        hap = fnd.t().contiguous().gather(0, src.long())                           # [n, c] = fnd[src, k]
        tmpl = fnd[:, 0]
        hap ^= (u > 1.0 - FLIP).to(torch.uint8)
        del u, src
        for a, b, core, carriers in plant:
            lo, hi = max(a, k0), min(b, k1)
            if lo < hi:
                hap[:, lo - k0:hi - k0] = torch.where(carriers[:, None], tmpl[None, lo - k0:hi - k0],
                                                      hap[:, lo - k0:hi - k0])
            if k0 <= core < k1:
                hap[:, core - k0] = carriers.to(torch.uint8)
        rows[k0:k1] = _pack_bits(hap.t().contiguous(), W)
    return rows


def _pack_bits(hap, W):
    """[c, n] 0/1 bytes -> int64 [c, W], haplotype h at bit h % 64 of word h // 64."""
    c, n = hap.shape
    full = torch.zeros((c, W * 64), dtype=torch.uint8, device=hap.device)
    full[:, :n] = hap
    v = full.view(torch.int64)                                # eight 0/1 bytes a word
    v = (v | (v >> 7)) & 0x0003000300030003
    v = (v | (v >> 14)) & 0x0000000F0000000F
    v = (v | (v >> 28)) & 0xFF
    return v.to(torch.uint8).view(torch.int64)


def _scan_inputs(case, seed):
    pos, gmap = _positions(case, seed)
    rows = _rows(case, seed, pos, gmap, case["nA"], case["founders"], case["sweeps"], 1)
    if case["nB"]:
        b = _rows(case, seed, pos, gmap, case["nB"], max(10, case["founders"] * 3 // 4), 0, 2)
        rows = torch.cat([rows, b], 1).contiguous()
    return rows, pos, gmap


def _params(case):
    opt = case.get("option", "")
    if opt == "crossing":
        return sg.selscan_default_params(include_crossing_term=1)
    if opt == "physical":
        return sg.selscan_default_params(use_physical_map=1)
    if opt == "cut10":
        return sg.selscan_default_params(ehh_cut=(1, 10))
    return sg.selscan_default_params()


def _aligned(nbytes):
    raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-raw.data_ptr()) % 256
    return raw[off:off + nbytes]


def _tick_cases(case):
    """The requests of a tick: samples between nA and nB haplotypes, marker
    counts around m, every third one an XPEHH request."""
    out = []
    for i in range(case["scans"]):
        f = i / max(1, case["scans"] - 1)
        n = int(round(case["nA"] * (case["nB"] / case["nA"]) ** f))
        m = int(case["m"] * (0.6 + 0.4 * ((i * 5) % 7) / 3.0))
        c = dict(case, nA=n, nB=0, m=m)
        if i % 3 == 2:
            c.update(nA=n // 2 + 1, nB=n // 2 + 3)
        out.append(c)
    return out


def _tick_scan(case, seed):
    rows, pos, gmap = _scan_inputs(case, seed)
    m, mode = case["m"], sg.MODE_XPEHH if case["nB"] else sg.MODE_IHS
    ipc, nd = (2, 6) if case["nB"] else (4, 4)
    f64 = dict(dtype=torch.float64, device="cuda")
    t = dict(status=torch.empty(m, dtype=torch.int8, device="cuda"),
             n1=torch.empty(m, dtype=torch.int32, device="cuda"), ihh_a=torch.empty(m, **f64),
             ihh_b=torch.empty(m, **f64), lnratio=torch.empty(m, **f64),
             stop=torch.empty((m, ipc), dtype=torch.int32, device="cuda"),
             digest=torch.empty((m, nd), dtype=torch.int64, device="cuda"),
             error=torch.zeros(1, dtype=torch.int32, device="cuda"))
    items = _aligned(sg.selscan_batch_item_bytes(m, mode))
    s = sg.selscan_scan()
    s.mode, s.nA, s.nB, s.m, s.ld, s.params = mode, case["nA"], case["nB"], m, rows.shape[1], _params(case)
    s.hap, s.pos_bp, s.gmap, s.items = rows.data_ptr(), pos.data_ptr(), gmap.data_ptr(), items.data_ptr()
    for f, v in t.items():
        setattr(s, f, v.data_ptr())
    return s, t, (rows, pos, gmap, items)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "normalize":
        g, m, n = _gen(seed, 5), case["m"], case["nA"]
        n1 = (n * torch.rand(m, generator=g, device="cuda") ** 2).to(torch.int32)
        u = torch.rand(m, generator=g, device="cuda")
        status = torch.where(torch.minimum(n1, n - n1) * 20 < n, 1, torch.where(u < 0.02, 3, 0)).to(torch.int8)
        score = torch.randn(m, generator=g, device="cuda", dtype=torch.float64) * 0.8 - 0.1
        score = torch.where(status == 0, score, float("nan"))      # as the scans leave it
        return dict(case=case, score=score, status=status, n1=n1)
    if kind == "pack":
        g, n, m = _gen(seed, 6), case["nA"], case["m"]
        shape = (n, m) if case["hap_major"] else (m, n)
        hap = torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.uint8)
        return dict(case=case, hap=hap)
    if kind == "tick":
        scans = [_tick_scan(c, seed + 31 * i) for i, c in enumerate(_tick_cases(case))]
        max_n = max(s.nA + s.nB for s, _, _ in scans)
        max_ld = max(s.ld for s, _, _ in scans)
        ws = _aligned(sg.selscan_batch_workspace_bytes(max_n, max_ld, len(scans), 256))
        return dict(case=case, scans=scans, max_n=max_n, max_ld=max_ld, ws=ws)
    if kind == "stream":
        sets = []
        for i in range(case["sets"]):
            sets.append(tuple(t.cpu().pin_memory() for t in _scan_inputs(case, seed + 31 * i)))
        return dict(case=case, sets=sets)
    rows, pos, gmap = _scan_inputs(case, seed)
    s = dict(case=case, rows=rows, pos=pos, gmap=gmap, params=_params(case), ws=None)
    if kind == "ehh":
        # a locus the report is asked for: common, away from the ends
        s["locus"] = case["m"] // 2 if case["sweeps"] else case["m"] // 3
    elif case["m"] >= 100_000:
        # a program that scans chromosomes one after another keeps the large workspace
        mode = sg.MODE_XPEHH if case["nB"] else sg.MODE_IHS
        s["ws"] = _aligned(sg.selscan_workspace_bytes(case["nA"] + case["nB"], case["m"], mode))
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "normalize":
        out = sg.selscan_normalize(state["score"], state["status"], state["n1"], case["nA"], case["bins"])
    elif kind == "pack":
        return sg.selscan_pack(state["hap"], case["nA"], hap_major=case["hap_major"])
    elif kind == "tick":
        scans = [s for s, _, _ in state["scans"]]
        for s in scans:
            sg.selscan_batch_prepare(s)
        sg.selscan_batch_run(scans, list(range(len(scans))), [0] * len(scans), [s.m for s in scans],
                             state["max_n"], state["max_ld"], state["ws"])
        for s in scans:
            sg.selscan_batch_finalize(s)
        return [t for _, t, _ in state["scans"]]
    elif kind == "stream":
        return [{f: t.clone() for f, t in r.items()}
                for r in sg_stream.scan_host_stream(state["sets"], sg.MODE_IHS, case["nA"])]
    elif kind == "ehh":
        out = sg.selscan_ehh(state["rows"], case["nA"], state["pos"], state["gmap"], state["locus"],
                             case["capacity"], params=state["params"])
    elif kind == "xpehh":
        out = sg.selscan_xpehh(state["rows"], case["nA"], case["nB"], state["pos"], state["gmap"],
                               params=state["params"], workspace=state["ws"])
    else:
        out = sg.selscan_ihs(state["rows"], case["nA"], state["pos"], state["gmap"],
                             params=state["params"], workspace=state["ws"])
    return {k: v for k, v in out.items() if not k.startswith("_")}


def _tick_or_sets(case):
    if case["kind"] == "tick":
        return _tick_cases(case)
    if case["kind"] == "stream":
        return [case] * case["sets"]
    return [case]


def work(case):
    """Inputs read once and outputs written once; the additions of the
    standardisation.  A scan's counts are integers: no floating-point work is
    claimed for them."""
    kind, n, m = case["kind"], case["nA"], case["m"]
    if kind == "normalize":
        return dict(bytes=m * (8 + 1 + 4 + 8) + case["bins"] * 24, flops=6 * m)
    if kind == "pack":
        return dict(bytes=m * n + m * 8 * ((n + 63) // 64), flops=0)
    if kind == "ehh":
        # the loci of six walks of about 100 steps, and the report
        return dict(bytes=6 * 100 * 8 * ((n + 63) // 64) + 16 * m + 6 * 8 * case["capacity"], flops=0)
    total = 0
    for c in _tick_or_sets(case):
        W = (c["nA"] + 63) // 64 + (c["nB"] + 63) // 64
        total += c["m"] * (8 * W + 16 + (61 if c["nB"] == 0 else 1 + 4 + 24 + 8 + 48))
    return dict(bytes=total, flops=0)


# ---------------------------------------------------------------- 64-bit values
def _unpack(rows, off, n):
    bits = torch.arange(64, device=rows.device)
    w = rows[:, off:off + (n + 63) // 64]
    return ((w[:, :, None] >> bits) & 1).reshape(rows.shape[0], -1)[:, :n].to(torch.int8)


class _Walks:
    """S(i) of every walk of a scan at once, from the definition: two
    haplotypes are one group over [core, x] when the sums of their alleles
    times random 64-bit numbers agree there (two different sequences agree
    with a chance of about 2^-64)."""

    def __init__(self, case, rows, pos, gmap):
        nA, nB = case["nA"], case["nB"]
        self.hap = _unpack(rows, 0, nA)
        if nB:
            self.hap = torch.cat([self.hap, _unpack(rows, (nA + 63) // 64, nB)], 1)
        m, n = self.hap.shape
        g = torch.Generator().manual_seed(12345)
        r = torch.randint(-(1 << 62), 1 << 62, (m,), generator=g, dtype=torch.int64).to(rows.device)
        self.h = torch.zeros((m + 1, n), dtype=torch.int64, device=rows.device)
        torch.cumsum(self.hap.long() * r[:, None], 0, out=self.h[1:])
        self.m, self.n, self.nA, self.nB = m, n, nA, nB
        self.pos, self.gmap = pos, gmap
        self.physical = case.get("option") == "physical"
        self.crossing = case.get("option") == "crossing"
        self.cut = 0.1 if case.get("option") == "cut10" else 0.05

    def counts(self, cores, xs):
        """[cores, classes] pair counts over the markers between each core and x."""
        lo, hi = torch.minimum(cores, xs), torch.maximum(cores, xs)
        key, idx = (self.h[hi + 1] - self.h[lo]).sort(1)
        if self.nB:
            lab = torch.stack([idx < self.nA, idx >= self.nA], 0)
        else:
            core = self.hap[cores].gather(1, idx) == 1
            lab = torch.stack([core, ~core], 0)
        t = torch.arange(self.n, device=key.device)
        new = torch.ones_like(key, dtype=torch.bool)
        new[:, 1:] = key[:, 1:] != key[:, :-1]
        start = torch.cummax(torch.where(new, t, 0), 1).values
        out = []
        for l in lab:
            before = torch.cumsum(l.long(), 1) - l.long()          # labelled haplotypes before t
            out.append(((before - before.gather(1, start)) * l).sum(1))
        out.append((t - start).sum(1))
        return torch.stack(out, 1)

    def walk(self, cores, direction):
        """(iHH [cores, 2], aborted [cores, walks]) of one direction."""
        dev, k = cores.device, cores.numel()
        if self.nB:
            D = torch.tensor([self.nA * (self.nA - 1) // 2, self.nB * (self.nB - 1) // 2,
                              self.n * (self.n - 1) // 2], device=dev).expand(k, 3)
            decide = [2, 2]
        else:
            n1 = self.hap[cores].long().sum(1)
            n0 = self.n - n1
            D = torch.stack([n1 * (n1 - 1) // 2, n0 * (n0 - 1) // 2, n1 * 0], 1)
            decide = [0, 1]
        ihh = torch.zeros((k, 2), dtype=torch.float64, device=dev)
        bad = torch.zeros((k, 2), dtype=torch.bool, device=dev)
        run_ = D[:, decide] > 0
        bad |= ~run_
        prev = torch.zeros((k, 3), dtype=torch.int64, device=dev)
        for s in range(0, k, 4096):
            prev[s:s + 4096] = self.counts(cores[s:s + 4096], cores[s:s + 4096])
        i = 1
        act = torch.arange(k, device=dev)
        while act.numel():
            x = cores[act] + direction * i
            out = (x < 0) | (x >= self.m)
            xc = x.clamp(0, self.m - 1)
            bp = (self.pos[xc] - self.pos[(xc - direction).clamp(0, self.m - 1)]).abs()
            out |= bp > 200_000
            bad[act[out]] |= run_[act[out]]
            run_[act[out]] = False
            act, xc, bp = act[~out], xc[~out], bp[~out]
            if not act.numel():
                break
            g = bp.double() if self.physical else (self.gmap[xc] - self.gmap[xc - direction]).abs()
            g = torch.where(bp > 20_000, g * (20_000.0 / bp.clamp(min=1).double()), g)
            per = max(1, 40_000_000 // self.n)
            S = torch.cat([self.counts(cores[act[s:s + per]], xc[s:s + per])
                           for s in range(0, act.numel(), per)])
            for w in (0, 1):
                ehh = S[:, decide[w]].double() / D[act, decide[w]].clamp(min=1).double()
                # a cutoff met exactly goes on: decided in integers
                stop = S[:, decide[w]] * round(1 / self.cut) < D[act, decide[w]]
                del ehh
                on = run_[act, w]
                add = on if self.crossing else on & ~stop
                term = (prev[act, w] + S[:, w]).double() * g / (2.0 * D[act, w].clamp(min=1).double())
                ihh[act, w] += torch.where(add, term, 0.0)
                run_[act, w] = on & ~stop
            prev[act] = S
            act = act[run_[act].any(1)]
            i += 1
        return ihh, bad


def _scan_exact(case, rows, pos, gmap):
    w = _Walks(case, rows, pos, gmap)
    n1 = w.hap.long().sum(1)
    keep = torch.ones(w.m, dtype=torch.bool, device=rows.device)
    if not case["nB"]:
        keep = torch.minimum(n1, w.n - n1) * 20 >= w.n
    cores = keep.nonzero()[:, 0]
    ihh = torch.zeros((w.m, 2), dtype=torch.float64, device=rows.device)
    bad = torch.zeros((w.m, 2), dtype=torch.bool, device=rows.device)
    for d in (-1, 1):
        a, b = w.walk(cores, d)
        ihh[cores] += a
        bad[cores] |= b
    ok = keep & ~bad.any(1) & (ihh > 0).all(1)
    ratio = torch.where(ok, torch.log(ihh[:, 0] / ihh[:, 1]), float("nan"))
    return ihh[:, 0], ihh[:, 1], ratio


def exact(case, seed):
    kind = case["kind"]
    if kind == "pack":
        return None                                   # bytes: equal or not
    if kind == "normalize":
        s = prepare(case, seed)
        n, nb = case["nA"], case["bins"]
        ok = s["status"] == 0
        b = (s["n1"].long() * nb // n).clamp(0, nb - 1)
        x, bb = s["score"][ok], b[ok]
        cnt = torch.bincount(bb, minlength=nb)
        nan = torch.full((nb,), float("nan"), dtype=torch.float64, device=x.device)
        mean, sd = nan.clone(), nan.clone()
        for q in range(nb):
            v = x[bb == q]
            if v.numel() >= 1:
                mean[q] = v.sum() / v.numel()
            if v.numel() >= 2:
                sd[q] = torch.sqrt(((v - mean[q]) ** 2).sum() / (v.numel() - 1))
        good = ok & (cnt[b] >= 2) & (sd[b] > 0)
        score = torch.where(good, (s["score"] - mean[b]) / sd[b], float("nan"))
        return dict(score=score, count=None, mean=mean, sd=sd)
    if kind == "tick":
        out = []
        if sum(c["m"] * (c["nA"] + c["nB"]) for c in _tick_cases(case)) > 40_000_000:
            return None
        for i, c in enumerate(_tick_cases(case)):
            a, b, r = _scan_exact(c, *_scan_inputs(c, seed + 31 * i))
            out.append(dict(ihh_a=a, ihh_b=b, lnratio=r))
        return out
    if kind == "stream" or case["m"] * (case["nA"] + case["nB"]) > 30_000_000:
        return None                                   # minutes in plain torch
    if kind == "ehh":
        s = prepare(case, seed)
        w = _Walks(case, s["rows"], s["pos"], s["gmap"])
        core = torch.tensor([s["locus"]], device="cuda")
        vals = torch.zeros((3, 2), dtype=torch.float64)
        for d, sign in enumerate((-1, 1)):
            ihh, _ = w.walk(core, sign)
            vals[0, d], vals[1, d] = ihh[0, 0], ihh[0, 1]
        # Eq. 1: the whole sample as one class
        whole = _Walks(dict(case, nB=0), s["rows"], s["pos"], s["gmap"])
        n = whole.n
        D = n * (n - 1) // 2
        for d, sign in enumerate((-1, 1)):
            S, i, acc = whole.counts(core, core)[0, 2].item(), 1, 0.0
            while True:
                x = s["locus"] + sign * i
                if x < 0 or x >= whole.m:
                    break
                bp = abs(int(s["pos"][x]) - int(s["pos"][x - sign]))
                if bp > 200_000:
                    break
                g = abs(float(s["gmap"][x]) - float(s["gmap"][x - sign]))
                g = g * (20_000.0 / bp) if bp > 20_000 else g
                T = whole.counts(core, torch.tensor([x], device="cuda"))[0, 2].item()
                if T * 20 < D:
                    break
                acc += (S + T) * g / (2.0 * D)
                S, i = T, i + 1
            vals[2, d] = acc
        return dict(ihh=vals.cuda())
    a, b, r = _scan_exact(case, *_scan_inputs(case, seed))
    if kind == "xpehh":
        return dict(ihhA=a, ihhB=b, lnratio=r)
    return dict(ihh1=a, ihh0=b, lnratio=r)
