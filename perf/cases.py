"""The workloads whose speed this library is judged by: what its users have it do,
through the public entry points, from one micro-batch to a megabase pair.

  listed()          the named cases
  draw(rng)         one more case of the same ranges
  prepare(case, s)  inputs made from seed s, parameters, outputs, handles
  run(state)        one pass, as a user's program makes it
  work(case)        bytes and operations one pass cannot do without
  exact(case, s)    what run() returns, computed plainly in 64 bits, where that is cheap

The recipes are those of the benchmark: short DNA pairs, protein pairs of uneven
length, noisy long reads, a serving mix's lengths, one megabase pair, edit-distance
pairs and structured RNAs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_06225_gb300 as F

DEV = "cuda"
RESULT_WORDS = F.RESULT_DTYPE.itemsize // 4
WORKSPACE = 96 << 30  # the long reads' traceback (about 77 GB) fits one wave
OPS_PER_CELL = 9      # affine cell update with its choice bits

_CTX = None


def _context():
    """The program's one context: its workspace serves every batch."""
    global _CTX
    if _CTX is None:
        _CTX = F.Context(0, WORKSPACE)
    return _CTX


# ---- cases -------------------------------------------------------------------

def listed():
    return [
        # a read mapper's candidate extensions: many short pairs, scores only
        dict(name="dna128_score", kind="align", gen="short", pairs=1000, lmin=128, lmax=128,
             err=0.05, mode="global", affine=1, band=-1, xdrop=-1, zdrop=-1, running=False,
             traceback=False),
        # a protein service's micro-batch: latency counts
        dict(name="protein_micro", kind="align", gen="protein", pairs=64, lmin=100, lmax=1000,
             err=0.02, mode="local", affine=1, band=-1, xdrop=-1, zdrop=-1, running=False,
             traceback=True),
        # all-against-all protein comparison: throughput over uneven lengths
        dict(name="protein_100k", kind="align", gen="protein", pairs=100_000, lmin=100, lmax=1000,
             err=0.02, mode="local", affine=1, band=-1, xdrop=-1, zdrop=-1, running=False,
             traceback=True),
        # the captured pipeline replayed for each batch of a steady stream
        dict(name="protein_graph", kind="graph", gen="protein", pairs=4096, lmin=100, lmax=1000,
             err=0.02, mode="local", affine=1, band=-1, xdrop=-1, zdrop=-1, running=False,
             traceback=True),
        # noisy long reads against their reference windows
        dict(name="long_reads_xdrop", kind="align", gen="reads", pairs=10_000, lmin=10_000,
             lmax=50_000, err=0.1, mode="global", affine=1, band=256, xdrop=400, zdrop=-1,
             running=False, traceback=True),
        # read extension that must survive long gaps
        dict(name="reads_zdrop", kind="align", gen="reads", pairs=1500, lmin=2000, lmax=6000,
             err=0.1, mode="global", affine=1, band=256, xdrop=-1, zdrop=400, running=False,
             traceback=True),
        # a serving batch of banded reads, log-normal lengths
        dict(name="reads_banded", kind="align", gen="lognormal", pairs=512, lmin=100, lmax=20_000,
             err=0.1, mode="global", affine=1, band=256, xdrop=-1, zdrop=-1, running=False,
             traceback=True),
        # one megabase pair with a 5 kb insertion: whole-contig comparison
        dict(name="pair_1mbp_xdrop", kind="long", length=1_000_000, err=0.01, seg=5000, mode="global",
             affine=1, band=-1, xdrop=1000, zdrop=-1, running=False, traceback=True),
        # the longest banded request of the serving mix, spread over the device
        dict(name="pair_80k_banded", kind="long", length=80_000, err=0.1, seg=0, mode="global",
             affine=1, band=256, xdrop=-1, zdrop=-1, running=False, traceback=True),
        # edit distance of similar sequences with the edits themselves
        dict(name="edit_4000", kind="search", pairs=8192, length=4000, err=0.05, alphabet=4, band=-1,
             adapt=False, traceback=True),
        # folding screens: every fold of a set of RNAs, exact and with X-drop
        dict(name="rna_300", kind="fold", seqs=1024, lmin=300, lmax=300, xdrop=-1, min_loop=3,
             traceback=True),
        dict(name="rna_500_xdrop", kind="fold", seqs=1024, lmin=500, lmax=500, xdrop=2, min_loop=3,
             traceback=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fam = rng.choice(["short", "protein", "protein", "graph", "reads", "reads", "lognormal", "mid",
                      "long_xdrop", "long_band", "search", "search", "fold", "fold"])
    tb = rng.random() < 0.75
    c = dict(kind="align", gen=fam, pairs=0, lmin=0, lmax=0, err=0.1, mode="global", affine=1, band=-1,
             xdrop=-1, zdrop=-1, running=False, traceback=tb)
    if fam == "short":
        c.update(pairs=_log(rng, 60, 40_000), lmin=rng.randint(40, 130), err=rng.choice([0.02, 0.05, 0.1]),
                 mode=rng.choice(["global", "global", "local"]), affine=rng.choice([1, 1, 0]))
        c.update(lmax=c["lmin"] + rng.randint(0, 170))
    elif fam in ("protein", "graph"):
        c.update(gen="protein", kind="graph" if fam == "graph" else "align", err=0.02,
                 pairs=_log(rng, 16, 8000 if fam == "graph" else 60_000), lmin=rng.randint(50, 150),
                 lmax=rng.randint(300, 1100), mode=rng.choice(["local", "local", "global"]),
                 affine=rng.choice([1, 1, 1, 0]))
    elif fam in ("reads", "mid"):
        c.update(gen="reads", pairs=_log(rng, 40, 4000), lmin=_log(rng, 500, 9000), err=rng.choice([0.05, 0.1]),
                 band=rng.choice([-1, 256, 256, 400]))
        c.update(lmax=c["lmin"] * rng.randint(2, 4))
        if fam == "mid":
            c.update(affine=2, xdrop=rng.randint(100, 400))
        else:
            t = rng.randint(80, 500)
            c.update(**({"zdrop": t} if rng.random() < 0.35 else {"xdrop": t}),
                     running=rng.random() < 0.25, mode=rng.choice(["global", "global", "local"]))
    elif fam == "lognormal":
        c.update(pairs=_log(rng, 8, 1500), lmin=100, lmax=_log(rng, 5000, 30_000), band=rng.randint(30, 300),
                 affine=rng.choice([1, 1, 0]))
    elif fam in ("long_xdrop", "long_band"):
        xd = fam == "long_xdrop"
        L = _log(rng, 90_000, 600_000) if xd else _log(rng, 8000, 120_000)
        for k in ("gen", "pairs", "lmin", "lmax"):
            c.pop(k)
        c.update(kind="long", length=L, seg=rng.choice([0, 500, 3000]) if xd else 0,
                 err=rng.choice([0.01, 0.05]), xdrop=rng.randint(300, 1200) if xd else -1,
                 band=-1 if xd else rng.randint(60, 400), traceback=True)
        if xd and c["seg"] == 3000:
            c["xdrop"] = rng.randint(6100, 7000)  # carries the alignment over the inserted segment
            c["length"] = min(L, 250_000)
    elif fam == "search":
        L = _log(rng, 300, 6000)
        e = rng.choice([0.01, 0.05, 0.1, 0.3])
        c = dict(kind="search", pairs=max(32, min(32_768, int(1.6e11 / (L * L * (e * e + 0.003))
                                                            * rng.uniform(0.02, 0.3)))), length=L, err=e,
                 alphabet=rng.choice([0, 4, 4]), band=rng.choice([-1, -1, 64]), adapt=rng.random() < 0.25,
                 traceback=tb)
    else:
        lo = _log(rng, 40, 1000)
        hi = lo + rng.randint(0, lo // 2)
        mean = (lo + hi) / 2
        c = dict(kind="fold", seqs=max(4, min(4096, int(5e11 / mean ** 3 * rng.uniform(0.02, 0.25)))), lmin=lo,
                 lmax=hi, xdrop=rng.choice([-1, -1, 2, 8]), min_loop=rng.choice([0, 3, 3]), traceback=tb)
    return c


# ---- inputs --------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _offsets(lens):
    off = torch.zeros_like(lens)
    off[1:] = torch.cumsum(lens, 0)[:-1]
    return off


def _geometric(n, p, g):
    """Geometric(p) on 1, 2, ..."""
    u = torch.rand(n, generator=g, device=DEV).clamp_min_(1e-12)
    return (torch.log(u) / math.log(1.0 - p)).floor_().to(torch.int64) + 1


def _mutate(ref, lens, p_sub, p_ins, p_del, geom, alphabet, fill, g):
    """Each residue of the concatenated `ref` draws at most one event:
    substitution, deletion of a run that starts there (within its sequence), or
    an insertion before it.  Returns (codes, lengths)."""
    n = ref.numel()
    ends = torch.cumsum(lens, 0)
    u = torch.rand(n, generator=g, device=DEV)
    is_del = (u >= p_sub) & (u < p_sub + p_del)
    is_ins = (u >= p_sub + p_del) & (u < p_sub + p_del + p_ins)
    shift = torch.randint(1, alphabet, (n,), generator=g, device=DEV, dtype=torch.uint8)
    base = torch.where(u < p_sub, (ref + shift) % alphabet, ref)
    del u, shift
    at = is_del.nonzero().flatten()
    run = _geometric(at.numel(), geom, g) if geom else torch.ones_like(at)
    stop = torch.minimum(at + run, ends[torch.searchsorted(ends, at, right=True)])
    diff = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    one = torch.ones_like(at, dtype=torch.int32)
    diff.index_add_(0, at, one).index_add_(0, stop, -one)
    keep = torch.cumsum(diff[:n], 0) <= 0
    del diff, is_del
    counts = keep.to(torch.int64)
    at = is_ins.nonzero().flatten()
    counts[at] += _geometric(at.numel(), geom, g) if geom else 1
    last = torch.cumsum(counts, 0)  # one past the slots of each residue
    out = fill(int(last[-1]))
    out[(last - 1)[keep]] = base[keep]
    upto = last[ends - 1]
    qlens = torch.diff(upto, prepend=torch.zeros(1, dtype=upto.dtype, device=DEV))
    return out, qlens


def _uniform(k, n, g):
    return torch.randint(0, k, (n,), generator=g, device=DEV, dtype=torch.uint8)


def _lengths(case, g):
    n, lo, hi = case["pairs"], case["lmin"], case["lmax"]
    if case["gen"] == "lognormal":  # the serving mix: median 2000, sigma 1
        x = torch.randn(n, generator=g, device=DEV).exp_() * 2000.0
        return x.round_().clamp_(lo, hi).to(torch.int64)
    return torch.randint(lo, hi + 1, (n,), generator=g, device=DEV)


def _protein_tables():
    rng = np.random.default_rng(2)
    s = np.triu(rng.integers(-4, 4, size=(20, 20)), 1)
    s = s + s.T
    np.fill_diagonal(s, rng.integers(4, 12, size=20))
    w = rng.uniform(1.0, 10.0, size=20)
    return s.astype(np.int8), np.cumsum(w / w.sum())


def _dna_table():
    s = np.full((4, 4), -4, np.int8)
    np.fill_diagonal(s, 2)
    return s


def _pairs(case, g):
    """(query codes, query lengths, reference codes, reference lengths)."""
    e = case["err"]
    if case.get("gen") == "protein":
        cdf = torch.tensor(_protein_tables()[1][:-1], dtype=torch.float32, device=DEV)

        def fill(n):
            return torch.bucketize(torch.rand(n, generator=g, device=DEV), cdf, right=True).to(torch.uint8)

        rl, ql = _lengths(case, g), _lengths(case, g)
        r, q = fill(int(rl.sum())), fill(int(ql.sum()))
        ident = torch.rand(case["pairs"], generator=g, device=DEV) * 0.4 + 0.3
        pair = torch.repeat_interleave(torch.arange(case["pairs"], device=DEV), ql)
        pos = torch.arange(q.numel(), device=DEV) - _offsets(ql)[pair]
        copy = (pos < rl[pair]) & (torch.rand(q.numel(), generator=g, device=DEV) < ident[pair])
        src = (_offsets(rl)[pair] + pos).clamp_(0, r.numel() - 1)
        q = torch.where(copy, r[src], q)
        q, ql = _mutate(q, ql, 0.0, e / 2, e / 2, 0.7, 20, fill, g)
        return q, ql, r, rl

    def fill(n):
        return _uniform(4, n, g)

    if case["kind"] == "long":
        rl = torch.tensor([case["length"]], device=DEV)
    elif case["kind"] == "search":
        rl = torch.full((case["pairs"],), case["length"], device=DEV, dtype=torch.int64)
    else:
        rl = _lengths(case, g)
    r = fill(int(rl.sum()))
    if case.get("gen") in ("reads", "lognormal") or (case["kind"] == "long" and case["seg"] == 0):
        # sequencing errors: mostly insertions, some deletions, few substitutions
        q, ql = _mutate(r, rl, 0.1 * e, 0.42 * e, 0.21 * e, 0.7, 4, fill, g)
    else:  # divergence: substitutions, insertions and deletions in equal parts
        q, ql = _mutate(r, rl, e / 3, e / 3, e / 3, None, 4, fill, g)
    if case["kind"] == "long" and case["seg"]:
        n = q.numel()
        at = int(torch.randint(n // 4, 3 * n // 4, (1,), generator=g, device=DEV))
        q = torch.cat([q[:at], fill(case["seg"]), q[at:]])
        ql = ql + case["seg"]
    return q, ql, r, rl


def _rna(case, g):
    """Structured RNAs: uniform ACGU with a hairpin stem planted about every 40
    bases (a segment and, a loop further on, its reverse complement)."""
    n = case["seqs"]
    lens = torch.randint(case["lmin"], case["lmax"] + 1, (n,), generator=g, device=DEV)
    width = case["lmax"]
    x = torch.randint(0, 4, (n, width), generator=g, device=DEV, dtype=torch.uint8)
    step = torch.arange(10, device=DEV)
    rows = torch.arange(n, device=DEV)[:, None].expand(n, 10)
    for _ in range(max(1, width // 40)):
        stem = torch.randint(4, 11, (n,), generator=g, device=DEV)
        loop = torch.randint(4, 41, (n,), generator=g, device=DEV)
        room = (lens - 2 * stem - loop).clamp_min(0)
        a = (torch.rand(n, generator=g, device=DEV) * (room + 1)).to(torch.int64)
        src = (a[:, None] + step).clamp_max(width - 1)
        dst = (a + 2 * stem + loop)[:, None] - 1 - step
        on = (step < stem[:, None]) & (lens >= 2 * stem + loop)[:, None]
        x[rows[on], dst[on]] = 3 - x[rows[on], src[on]]
    keep = torch.arange(width, device=DEV) < lens[:, None]
    return x[keep], lens


def _cigar_room(case):
    """Ops for any CIGARs of the case's sizes: a program reserves its largest
    batch once.  Queries exceed their references' lengths by their insertions."""
    longest = case["length"] + case.get("seg", 0) if "length" in case else case["lmax"]
    return case.get("pairs", 1) * (2 * longest + longest // 4 + 64)


# ---- prepare and run -------------------------------------------------------------

def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    g = _gen(seed)
    ctx = _context()
    if case["kind"] == "fold":
        seq, lens = _rna(case, g)
        n = case["seqs"]
        return dict(case=case, ctx=ctx, n=n, seq=seq, off=_offsets(lens), lens=lens.to(torch.int32),
                    params=F.make_fold_params(min_loop=case["min_loop"],
                                              xdrop=None if case["xdrop"] < 0 else case["xdrop"],
                                              traceback=case["traceback"]),
                    out=torch.zeros(n * F.FOLD_RESULT_DTYPE.itemsize // 4, dtype=torch.int32, device=DEV),
                    partner=torch.zeros(n * case["lmax"], dtype=torch.int32, device=DEV))
    q, ql, r, rl = _pairs(case, g)
    n = int(ql.numel())
    tb = case["traceback"]
    cap = _cigar_room(case) if tb else 0
    s = dict(case=case, ctx=ctx, n=n, q=q, r=r, M=int(ql[0]), N=int(rl[0]), q_off=_offsets(ql),
             r_off=_offsets(rl), q_len=ql.to(torch.int32), r_len=rl.to(torch.int32), cap=cap,
             out=torch.zeros((n, RESULT_WORDS), dtype=torch.int32, device=DEV),
             cigar=torch.zeros(max(cap, 1), dtype=torch.int32, device=DEV))
    if case["kind"] == "search":
        s["params"] = F.make_search_params(traceback=tb, band=None if case["band"] < 0 else case["band"],
                                           adapt=(10, 50) if case["adapt"] else None,
                                           alphabet=case["alphabet"])
        return s
    protein = case.get("gen") == "protein"
    s["params"] = F.make_params(
        _protein_tables()[0] if protein else _dna_table(), mode=case["mode"], affine=case["affine"] != 0,
        mid=case["affine"] == 2, gap_open=11 if protein else 4,
        gap_extend=(1 if protein else 2) if case["affine"] else 4,
        band=None if case["band"] < 0 else case["band"], xdrop=None if case["xdrop"] < 0 else case["xdrop"],
        zdrop=None if case["zdrop"] < 0 else case["zdrop"], xdrop_running=case["running"], traceback=tb)
    if case["kind"] == "graph":
        longest = case["lmax"] + case["lmax"] // 5 + 16  # room for the queries' insertions
        bits = case["pairs"] * (longest // 2) * longest if tb else 0
        s["graph"] = F.Graph(ctx, s["params"], case["pairs"], longest, (2 << 30) + bits)
    return s


def run(s):
    kind = s["case"]["kind"]
    ctx = s["ctx"]
    if kind == "fold":
        F.check(ctx.fold_batch_ptr(s["params"], s["n"], s["seq"].data_ptr(), s["off"].data_ptr(),
                                   s["lens"].data_ptr(), s["out"].data_ptr(),
                                   s["partner"].data_ptr() if s["case"]["traceback"] else None, _stream()))
        words = s["out"].view(s["n"], -1)
        return {"score": words[:, 0], "rest": words[:, 1:], "partner": s["partner"]}
    cig = s["cigar"].data_ptr() if s["cap"] else None
    if kind == "long":
        F.check(ctx.align_long_ptr(s["params"], s["q"].data_ptr(), s["M"], s["r"].data_ptr(), s["N"],
                                   s["out"].data_ptr(), cig, s["cap"], _stream()))
    else:
        batch = (s["n"], s["q"].data_ptr(), s["q_off"].data_ptr(), s["q_len"].data_ptr(), s["r"].data_ptr(),
                 s["r_off"].data_ptr(), s["r_len"].data_ptr(), s["out"].data_ptr(), cig, s["cap"], _stream())
        if kind == "graph":
            F.check(s["graph"].launch_ptr(*batch))
        elif kind == "search":
            F.check(ctx.search_batch_ptr(s["params"], *batch))
        else:
            F.check(ctx.align_batch_ptr(s["params"], *batch))
    return {"score": s["out"][:, 0], "rest": s["out"][:, 1:], "cigar": s["cigar"]}


# ---- what a pass cannot do without -------------------------------------------------

def work(case):
    k = case["kind"]
    if k == "fold":
        n, L = case["seqs"], (case["lmin"] + case["lmax"]) / 2
        # every split term is an add and a max; each base read, its partner written
        return dict(bytes=n * (L * (5 if case["traceback"] else 1) + 36), flops=n * L ** 3 / 3)
    if k == "search":
        n, L, d = case["pairs"], case["length"], case["length"] * case["err"]
        width = d if case["band"] < 0 else min(d, 2 * case["band"])
        # a wavefront entry: three terms, their maximum, and its compared residues
        return dict(bytes=n * (2 * L + 72 + (4 * d if case["traceback"] else 0)), flops=n * (6 * d * width + 2 * L))
    if k == "long":
        n, L = 1, float(case["length"])
    elif case["gen"] == "lognormal":
        n, L = case["pairs"], min(3300.0, case["lmax"] / 2)
    else:
        n, L = case["pairs"], (case["lmin"] + case["lmax"]) / 2
    cells = L * L
    if case["band"] >= 0:
        cells = min(cells, L * (2 * case["band"] + 1))
    if max(case["xdrop"], case["zdrop"]) >= 0:  # live cells of an antidiagonal: gaps down to the threshold
        cells = min(cells, 2 * L * max(8.0, (max(case["xdrop"], case["zdrop"]) - 4) / 2))
    tb = case["traceback"]
    gaps = 0.2 if case.get("gen") != "short" else 0.1  # CIGAR ops per residue
    return dict(bytes=n * (2 * L + 72 + (4 * gaps * L if tb else 0)), flops=n * cells * OPS_PER_CELL)


# ---- plain 64-bit values -------------------------------------------------------------

def _exact_global_scores(case, seed):
    """Affine global scores of every pair, row by row over the whole batch."""
    q, ql, r, rl = (t.cpu().numpy() for t in _pairs(case, _gen(seed)))
    n, M, N = len(ql), int(ql.max()), int(rl.max())
    Q, R = np.zeros((n, M), np.int64), np.zeros((n, N), np.int64)
    Q[np.arange(M) < ql[:, None]] = q
    R[np.arange(N) < rl[:, None]] = r
    sub = (_protein_tables()[0] if case["gen"] == "protein" else _dna_table()).astype(np.int64)
    o, e = (11, 1) if case["gen"] == "protein" else (4, 2)
    j = np.arange(N + 1)
    low = -(1 << 40)
    H = np.broadcast_to(np.where(j > 0, -(o + e * j), 0), (n, N + 1)).copy()
    V = np.full((n, N + 1), low)
    score = np.where(ql == 0, H[np.arange(n), rl], 0)
    for i in range(1, M + 1):
        V = np.maximum(V, H - o) - e
        best = V.copy()
        best[:, 1:] = np.maximum(best[:, 1:], H[:, :-1] + sub[Q[:, i - 1][:, None], R])
        # horizontal gaps: the best of the cells to the left, less open and extend
        run = np.maximum.accumulate(best + e * j, axis=1)
        H = best.copy()
        H[:, 1:] = np.maximum(best[:, 1:], run[:, :-1] - o - e * j[1:])
        score = np.where(ql == i, H[np.arange(n), rl], score)
    return score


def _exact_fold_scores(case, seed):
    """Most nested base pairs of each RNA, span by span over the whole batch."""
    seq, lens = _rna(case, _gen(seed))
    n, L = case["seqs"], int(lens.max())
    x = torch.zeros((n, L), dtype=torch.int64, device=DEV)
    x[torch.arange(L, device=DEV) < lens[:, None]] = seq.to(torch.int64)
    tab = torch.zeros((n, L + 1, L), dtype=torch.int64, device=DEV)  # tab[:, k, i] = F(i, i + k - 1); row 0 empty
    score = torch.zeros(n, dtype=torch.int64, device=DEV)
    for k in range(1, L):
        w = L - k
        best = torch.zeros((n, w), dtype=torch.int64, device=DEV)
        if k - 1 >= case["min_loop"]:
            a, b = x[:, :w], x[:, k:]
            pair = (a + b == 3) | ((a + b == 5) & (a != b))
            best = torch.where(pair, tab[:, k - 1, 1:w + 1] + 1, best)
        for t in range(1, k + 1):
            best = torch.maximum(best, tab[:, t, :w] + tab[:, k + 1 - t, t:t + w])
        tab[:, k + 1, :w] = best
        score = torch.where(lens == k + 1, best[:, 0], score)
    return score


def exact(case, seed):
    if case["kind"] == "fold" and case["xdrop"] < 0 and case["lmax"] <= 320 and case["seqs"] <= 1100:
        return {"score": _exact_fold_scores(case, seed), "rest": None, "partner": None}
    if (case["kind"] == "align" and case["gen"] in ("short", "protein") and case["mode"] == "global"
            and case["affine"] == 1 and case["pairs"] * case["lmax"] ** 2 < 2e8):
        return {"score": _exact_global_scores(case, seed), "rest": None, "cigar": None}
    return None
