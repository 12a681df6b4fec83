"""Edges of the antidiagonal sweep and of the warp walks, against the oracle, bit for
bit: windows that move several times in one pair and in both directions, at every group
width; blocks of antidiagonals that alternate between the checked and the unchecked form
(the live range touches the band and leaves it again) for compared and looked-up scores;
paths that leave the walk's eight diagonals by long gaps both ways."""
import functools

import numpy as np
import pytest

import synth
from gpu_util import compare, oracle_batch

pytestmark = pytest.mark.gpu

DNA_S = synth.dna_subst(2, -4)
PROT_S = synth.protein_subst(np.random.default_rng(2))


@pytest.fixture(scope="module")
def F():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_06225_gb300 as F

    return F


@pytest.fixture(scope="module")
def ctx(F):
    c = F.Context(0, 24 << 30)
    yield c
    F.lib().filtr_test_set_first_width(c.handle, 0)
    F.lib().filtr_test_set_packed_sweep(c.handle, 0)
    c.close()


def gapped(rng, alphabet, between, gaps):
    """(query, reference): `between` common residues, then a gap, and so on; a positive
    gap inserts that many residues into the query, a negative one leaves residues of
    the reference out of it."""
    q, r = [], []
    for g in list(gaps) + [0]:
        core = rng.integers(0, alphabet, between).astype(np.uint8)
        extra = rng.integers(0, alphabet, abs(g)).astype(np.uint8)
        q += [core, extra] if g > 0 else [core]
        r += [core, extra] if g < 0 else [core]
    return np.concatenate(q), np.concatenate(r)


@functools.lru_cache(maxsize=1)
def drifting(W, alphabet):
    """Gaps of one sign until the live range has left a window of 256 W slots (two
    diagonals each) that stayed, twice as many back, and again; and the oracle's results."""
    rng = np.random.default_rng(100 + W + alphabet)
    n = max(6, 512 * W * 5 // (4 * 150) + 2)
    ways = [150] * n + [-150] * (2 * n) + [150] * n
    pairs = [gapped(rng, alphabet, 180, w) for w in (ways, [-g for g in ways])]
    o, e, x = (4, 2, 380) if alphabet == 4 else (11, 1, 250)
    b = synth.pack([p[0] for p in pairs], [p[1] for p in pairs], alphabet, DNA_S if alphabet == 4 else PROT_S)
    sc = dict(mode="global", affine=True, gap_open=o, gap_extend=e, xdrop=x, traceback=True)
    return b, sc, oracle_batch(b, sc)


@pytest.mark.parametrize("packed", [0, 1])
@pytest.mark.parametrize("W", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("alphabet", [4, 20])
def test_window_moves_both_ways(F, ctx, packed, W, alphabet):
    """A first group width of W warps under X-drop, both cell widths."""
    b, sc, want = drifting(W, alphabet)
    assert F.lib().filtr_test_set_first_width(ctx.handle, W) == F.OK
    assert F.lib().filtr_test_set_packed_sweep(ctx.handle, packed) == F.OK
    try:
        res, cig, rc = F.align_batch(ctx, F.make_params(b.subst, **sc), b)
        assert rc == 0, F.last_error()
        compare(b, sc, res, cig, *want, label=f"W={W}")
    finally:
        F.lib().filtr_test_set_first_width(ctx.handle, 0)
        F.lib().filtr_test_set_packed_sweep(ctx.handle, 0)
    assert (res["status"] == 0).all()  # the gaps were carried: the path went all the way


@pytest.mark.parametrize("mode", ["global", "local"])
@pytest.mark.parametrize("alphabet", [4, 20])
@pytest.mark.parametrize("drop", [dict(xdrop=150), dict(xdrop=150, xdrop_running=True), dict(zdrop=150)])
@pytest.mark.parametrize("W", [1, 2, 4, 8])
def test_checked_and_unchecked_blocks(F, ctx, W, drop, alphabet, mode):
    """Drifts of 40 to 110 diagonals under a literal band of 100: blocks at the band, past
    it and away from it; lengths between cover every offset within 16 antidiagonals."""
    rng = np.random.default_rng(200 + W + alphabet)
    qs, rs = [], []
    for t in range(24):
        gaps = [int(g) for g in rng.integers(20, 56, 2)]
        q, r = gapped(rng, alphabet, 170 + t, [gaps[0], gaps[1], -gaps[0], -gaps[1], -gaps[1], -gaps[0], gaps[0], gaps[1]])
        qs.append(q)
        rs.append(r[:len(r) - t % 7])
    b = synth.pack(qs, rs, alphabet, DNA_S if alphabet == 4 else PROT_S)
    o, e = (4, 2) if alphabet == 4 else (11, 1)
    sc = dict(mode=mode, affine=True, gap_open=o, gap_extend=e, band=100, band_literal=True, traceback=True, **drop)
    assert F.lib().filtr_test_set_first_width(ctx.handle, W) == F.OK
    try:
        res, cig, rc = F.align_batch(ctx, F.make_params(b.subst, **sc), b)
        assert rc == 0, F.last_error()
        compare(b, sc, res, cig, *oracle_batch(b, sc), label=f"W={W}")
    finally:
        F.lib().filtr_test_set_first_width(ctx.handle, 0)


LONG_GAPS = [7, -7, 8, -8, 9, 31, -31, 32, -33, 64, -64, 96, -97, 33, -32, -9, 150, -150, 1, -1, 2, -2]


@pytest.mark.parametrize("alphabet", [4, 20])
@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(band=260), dict(xdrop=400), dict(affine=False),
                                dict(mode="local"), dict(mode="local", band=260)])
def test_walk_across_long_gaps(F, ctx, kw, alphabet):
    """Gaps around the walk's window (eight diagonals by 32 rows) in both directions, with
    few and many residues between them, in every layout that a warp walks."""
    rng = np.random.default_rng(300 + alphabet)
    qs, rs = [], []
    for between in (40, 70, 100, 133):
        for sign in (1, -1):
            q, r = gapped(rng, alphabet, between, [sign * g for g in LONG_GAPS])
            qs.append(q)
            rs.append(r)
    b = synth.pack(qs, rs, alphabet, DNA_S if alphabet == 4 else PROT_S)
    o, e = (4, 2) if alphabet == 4 else (11, 1)
    sc = dict(dict(mode="global", affine=True, gap_open=o, gap_extend=e, traceback=True), **kw)
    if sc.get("affine") is False:
        sc.pop("gap_open")
    res, cig, rc = F.align_batch(ctx, F.make_params(b.subst, **sc), b)
    assert rc == 0, F.last_error()
    osc = {k: v for k, v in sc.items() if k != "precision"}
    compare(b, osc, res, cig, *oracle_batch(b, osc), label=str(kw))


@pytest.mark.parametrize("mode", ["global", "local"])
@pytest.mark.parametrize("drop", [dict(xdrop=60), dict(zdrop=60), dict(xdrop=60, band=80)])
@pytest.mark.parametrize("W", [1, 2, 4])
def test_one_match_score_over_twenty_letters(F, ctx, W, drop, mode):
    """A protein matrix with one match and one mismatch score, which the sweep may not
    treat as DNA: its codes do not fit two bits.  Mutations move codes by four, eight,
    twelve and sixteen, so that any comparison of low bits alone takes them for matches."""
    rng = np.random.default_rng(400 + W)
    subst = np.full((20, 20), -3, np.int8)
    np.fill_diagonal(subst, 4)
    qs, rs = [], []
    for n in (1, 17, 90, 300, 700, 1500):
        r = rng.integers(0, 20, n).astype(np.uint8)
        q = np.where(rng.random(n) < 0.15, (r + 4 * rng.integers(1, 5, n)) % 20, r).astype(np.uint8)
        qs.append(np.concatenate([q[:n // 2], rng.integers(0, 20, n // 60).astype(np.uint8), q[n // 2:]]))
        rs.append(r)
    b = synth.pack(qs, rs, 20, subst)
    sc = dict(mode=mode, affine=True, gap_open=5, gap_extend=2, traceback=True, **drop)
    assert F.lib().filtr_test_set_first_width(ctx.handle, W) == F.OK
    try:
        res, cig, rc = F.align_batch(ctx, F.make_params(b.subst, **sc), b)
        assert rc == 0, F.last_error()
        compare(b, sc, res, cig, *oracle_batch(b, sc), label=f"W={W}")
    finally:
        F.lib().filtr_test_set_first_width(ctx.handle, 0)


@pytest.mark.parametrize("mode", ["local", "global"])
@pytest.mark.parametrize("long", [False, True])
def test_regions_as_wide_as_the_widest_window(F, ctx, mode, long):
    """Antidiagonals of up to 8192 live cells, the documented limit, where nothing is
    pruned; 8193 are too many.  The longer side makes the range move off the window's
    middle.  Batches and the checkpointed sweep, both cell widths."""
    rng = np.random.default_rng(500)
    qs, rs = [], []
    for m, n in [(8140, 8500), (8170, 8600), (8900, 8180), (8187, 8400), (8300, 8191), (8191, 8191), (8192, 8192)]:
        r = rng.integers(0, 4, n).astype(np.uint8)
        q = np.where(rng.random(n) < 0.1, rng.integers(0, 4, n), r).astype(np.uint8)
        qs.append(np.concatenate([q, rng.integers(0, 4, m).astype(np.uint8)])[:m])
        rs.append(r)
    # (a global corner-to-corner band of free gaps keeps all cells: no gap costs anything)
    sc = dict(mode=mode, affine=True, gap_open=4 if mode == "local" else 0, gap_extend=2 if mode == "local" else 0,
              xdrop=7999, traceback=True)
    b = synth.pack(qs, rs, 4, synth.dna_subst(0 if mode == "global" else 1, -1))
    params = F.make_params(b.subst, **sc)
    out = []
    for packed in (0, 1):
        assert F.lib().filtr_test_set_packed_sweep(ctx.handle, packed) == F.OK
        if long:
            F.lib().filtr_test_set_checkpoint(ctx.handle, 4096)
        try:
            if long:
                got = [F.align_long(ctx, params, q, r) for q, r in zip(qs, rs)]
                res, cig = np.array([g[0] for g in got]), np.concatenate([g[1] for g in got])
            else:
                res, cig, rc = F.align_batch(ctx, params, b)
                assert rc == 0, F.last_error()
                cig = cig[:int(res["cigar_len"].sum())]
                # (ranges of 8191 and 8192 cells that move may need the int32 sweep's window)
                assert ctx.last_stats()["pairs_xd16_rerun"] <= 2
        finally:
            F.lib().filtr_test_set_packed_sweep(ctx.handle, 0)
            F.lib().filtr_test_set_checkpoint(ctx.handle, 0)
        assert list(res["status"]) == [0] * 6 + [4]
        out.append((res[:-1].tobytes(), cig.tobytes()))
    assert out[0] == out[1]
