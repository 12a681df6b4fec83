"""Tiled pairs with a warp per row strip (k_split.cuh) against the warp-per-pair
kernels and the oracle, bit for bit: strip edges (256 and 512 rows), references
from 1 column, bands whose strips start past the first column or hold no cell,
pairs of very uneven height in one queue, both planners, the captured pipeline,
and workspaces that leave no room for the hand-over slots."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

DNA_S = synth.dna_subst(2, -4)
PROT_S = synth.protein_subst(np.random.default_rng(2))
ROWS = [1, 255, 256, 257, 511, 512, 513, 769, 1024, 1025, 1300]
COLS = [1, 2, 31, 32, 33, 63, 64, 65, 300, 700]


@pytest.fixture(scope="module")
def F():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_06225_gb300 as F

    return F


@pytest.fixture(scope="module")
def ctx(F):
    c = F.Context(0, 8 << 30)
    yield c
    F.lib().filtr_test_set_split(c.handle, 0)
    c.close()


def pairs(alphabet, seed, sizes):
    rng = np.random.default_rng(seed)
    qs, rs = [], []
    for m, n in sizes:
        r = rng.integers(0, alphabet, n).astype(np.uint8)
        q = synth.mutate(rng, r, 0.1, 0.05, 0.05, 0.7, alphabet)[:m]
        qs.append(np.concatenate([q, rng.integers(0, alphabet, m - len(q)).astype(np.uint8)]))
        rs.append(r)
    return synth.pack(qs, rs, alphabet, DNA_S if alphabet == 4 else PROT_S)


def run(F, ctx, b, sc, mode, **kw):
    assert F.lib().filtr_test_set_split(ctx.handle, mode) == F.OK
    res, cig, rc = F.align_batch(ctx, F.make_params(b.subst, **sc), b, **kw)
    assert rc == 0, F.last_error()
    n = int(res["cigar_len"].sum()) if sc.get("traceback") else 0
    return res, cig[:n]


def same(a, b):
    assert a[0].tobytes() == b[0].tobytes()
    assert np.array_equal(a[1], b[1])


KINDS = {
    "global": dict(mode="global"),
    "local": dict(mode="local"),
    "global_linear": dict(mode="global", affine=False),
    "local_linear": dict(mode="local", affine=False),
    "band": dict(mode="global", band=20),
    "band_local": dict(mode="local", band=40),
    "band_literal": dict(mode="global", band=300, band_literal=True),
    "int32": dict(mode="global", precision=1),
}


@pytest.mark.parametrize("alphabet", [4, 20])
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("kind", list(KINDS))
def test_edges(F, ctx, kind, tb, alphabet):
    sc = dict(dict(affine=True, gap_open=11 if alphabet == 20 else 4, gap_extend=2), **KINDS[kind],
              traceback=tb)
    b = pairs(alphabet, 5, [(m, n) for m in ROWS for n in COLS])
    got = run(F, ctx, b, sc, 2)
    same(got, run(F, ctx, b, sc, 1))
    pick = list(range(0, b.n, 7))
    osc = {k: v for k, v in sc.items() if k != "precision"}
    ores = oracle.align_batch(b.subset(pick), **osc)[0]
    assert np.array_equal(got[0]["score"][pick].astype(np.int64), ores["score"])
    assert np.array_equal(got[0]["cells"][pick].astype(np.int64), ores["cells"])


@pytest.mark.parametrize("n", [1, 2, 300, 700])
@pytest.mark.parametrize("kind", ["local", "band"])
def test_uneven_heights(F, ctx, n, kind):
    """One tall pair among short ones; host (n < 256) and device plans, and both
    packed strip heights."""
    rng = np.random.default_rng(n)
    sizes = [(6000, 5500)] + [(int(rng.integers(1, 900)), int(rng.integers(1, 900))) for _ in range(n - 1)]
    sc = dict(dict(affine=True, gap_open=4, gap_extend=2, traceback=True), **KINDS[kind])
    b = pairs(4, 6, sizes)
    same(run(F, ctx, b, sc, 2), run(F, ctx, b, sc, 1))


def test_both_widths(F, ctx):
    """Pairs whose scores fit 15 bits beside pairs whose do not: two queues; the
    tall ones have more strips than a warp has lanes."""
    b = pairs(20, 7, [(700, 800)] * 5 + [(9000, 6000)] * 2 + [(300, 5000)] * 3)
    sc = dict(mode="local", affine=True, gap_open=11, gap_extend=1, traceback=True)
    same(run(F, ctx, b, sc, 2), run(F, ctx, b, sc, 1))


@pytest.mark.parametrize("sc", [dict(mode="global", precision=1), dict(mode="local"),
                                dict(mode="global", band=3000)])
def test_many_strips_at_once(F, ctx, sc):
    """One pair of 80 strips, all of them waiting in line from the start."""
    sc = dict(dict(affine=True, gap_open=4, gap_extend=2, traceback=True), **sc)
    b = pairs(4, 10, [(20400, 1500)])
    same(run(F, ctx, b, sc, 2), run(F, ctx, b, sc, 1))


def test_small_workspace(F):
    """No room for the slots, or only for less traceback: the warp-per-pair form."""
    b = pairs(4, 8, [(1100, 1000)] * 40)
    sc = dict(mode="local", affine=True, gap_open=4, gap_extend=2, traceback=True)
    big = F.Context(0, 1 << 30)
    want = run(F, big, b, sc, 1)
    big.close()
    for ws in (3 << 20, 8 << 20, 24 << 20, 40 << 20):
        small = F.Context(0, ws)
        try:
            same(run(F, small, b, sc, 2), want)
        finally:
            small.close()


@pytest.mark.parametrize("kind", ["local", "band", "global"])
def test_graph(F, ctx, kind):
    sc = dict(dict(affine=True, gap_open=4, gap_extend=2, traceback=True), **KINDS[kind])
    for n, room in ((40, 1 << 30), (900, 2 << 30)):
        rng = np.random.default_rng(n)
        b = pairs(4, 9, [(int(rng.integers(0, 1000)), int(rng.integers(0, 1000))) for _ in range(n)])
        want = run(F, ctx, b, sc, 1)
        for mode in (0, 2):
            F.lib().filtr_test_set_split(ctx.handle, mode)
            g = F.Graph(ctx, F.make_params(b.subst, **sc), n + 3, 1000, room)
            for _ in range(2):
                res, cig, st = F.graph_align(g, b)
                assert st == F.OK
                same((res, cig[:int(res["cigar_len"].sum())]), want)
            sub = b.subset([n // 2])
            res, cig, st = F.graph_align(g, sub)
            same((res, cig[:int(res["cigar_len"].sum())]), run(F, ctx, sub, sc, 1))
            g.close()


def test_tall_pair_in_a_batch(F, ctx):
    """300 unbanded pairs of a few hundred rows and one of 5000: the default rule
    plans them again, a warp per strip."""
    rng = np.random.default_rng(11)
    sizes = [(5000, 4000)] + [(int(rng.integers(100, 400)), int(rng.integers(100, 400))) for _ in range(300)]
    sc = dict(mode="local", affine=True, gap_open=11, gap_extend=1, traceback=True)
    b = pairs(20, 12, sizes)
    got = run(F, ctx, b, sc, 0)
    assert ctx.last_stats()["device_plan"] == 0
    same(got, run(F, ctx, b, sc, 1))


@pytest.mark.parametrize("mode,gaps", [("global", dict(affine=True, gap_open=4, gap_extend=2)),
                                       ("global", dict(affine=False, gap_extend=3)),
                                       ("local", dict(affine=True, gap_open=11, gap_extend=1))])
@pytest.mark.parametrize("band,literal", [(0, False), (3, False), (40, True), (300, False)])
def test_long_banded_low_strips(F, ctx, mode, gaps, band, literal):
    """One banded pair in strips of 128 rows: heights at the edges of one, two and
    five strips, bands narrower and wider than a strip."""
    for m, n in [(1, 1), (4, 60), (127, 127), (128, 140), (129, 100), (257, 257), (640, 650), (641, 641)]:
        b = pairs(4, 900 + m, [(m, n)])
        q, r = b.pair(0)
        sc = dict(mode=mode, traceback=True, band=band, band_literal=literal, **gaps)
        res, cig, rc = F.align_long(ctx, F.make_params(DNA_S, **sc), q, r)
        assert rc == 0, F.last_error()
        o = oracle.align(q, r, DNA_S, **sc)
        for f in ("score", "q_begin", "r_begin", "q_end", "r_end", "status", "cells"):
            assert int(res[f]) == int(o[f]), (m, n, f, int(res[f]), int(o[f]))
        assert np.array_equal(cig, o["cigar"]), (m, n)


def test_long_banded_either_height(F):
    """A workspace that holds the traceback of 256-row strips but not of 128-row ones."""
    b = pairs(4, 77, [(20000, 20000)])
    q, r = b.pair(0)
    prm = F.make_params(DNA_S, mode="global", affine=True, gap_open=4, gap_extend=2, band=64,
                        traceback=True)
    out = []
    for ws in (64 << 20, 5 << 20):  # the two heights need 5.9 and 4.3 MB
        c = F.Context(0, ws)
        try:
            res, cig, rc = F.align_long(c, prm, q, r)
            assert rc == 0, F.last_error()
            out.append((res.tobytes(), cig.tobytes()))
        finally:
            c.close()
    assert out[0] == out[1]


@pytest.mark.parametrize("n", [255, 256, 300])
def test_banded_batch_with_tall_pairs(F, ctx, n):
    """The default choice around the size where batches are planned on the device:
    many low banded pairs and a few tall ones, against the warp-per-pair kernels."""
    rng = np.random.default_rng(n)
    sizes = [(int(m), int(m) + 5) for m in rng.integers(40, 300, n - 3)] + [(3000, 2990), (2050, 2100), (1409, 1400)]
    b = pairs(4, 31 + n, sizes)
    sc = dict(mode="global", affine=True, gap_open=4, gap_extend=2, band=50, traceback=True)
    same(run(F, ctx, b, sc, 0), run(F, ctx, b, sc, 1))


@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("kind", ["local", "band"])
def test_tall_pair_without_room_for_strips(F, kind, tb):
    """A tall pair in a batch whose hand-over slots (301 pairs x 2 slots of 4001 words,
    19.3 MB) exceed a quarter of the workspace: the device's plan, whose shapes run
    side by side, is kept, and with room for the slots it is given up."""
    rng = np.random.default_rng(13)
    sizes = [(5000, 4000)] + [(int(rng.integers(100, 400)), int(rng.integers(100, 400))) for _ in range(300)]
    sc = dict(dict(affine=True, gap_open=11, gap_extend=1, traceback=tb), **KINDS[kind])
    b = pairs(20, 14, sizes)
    out = []
    for ws, planned_on_device in ((64 << 20, 1), (256 << 20, 0)):
        c = F.Context(0, ws)
        try:
            out.append(run(F, c, b, sc, 0))
            assert c.last_stats()["device_plan"] == planned_on_device
            same(out[-1], run(F, c, b, sc, 1))
        finally:
            c.close()
    same(out[0], out[1])


def strip_rows(F, ctx):
    import ctypes as C

    rows = C.c_int32(-1)
    assert F.lib().filtr_test_last_strip_rows(ctx.handle, C.byref(rows)) == F.OK
    return rows.value


@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("mode,gaps", [("global", dict(affine=True, gap_open=4, gap_extend=2)),
                                       ("global", dict(affine=False, gap_extend=3)),
                                       ("local", dict(affine=True, gap_open=11, gap_extend=1)),
                                       ("local", dict(affine=False, gap_extend=5))])
@pytest.mark.parametrize("band,literal", [(0, False), (3, False), (40, True), (300, False)])
def test_long_pair_in_strips_of_128_rows(F, ctx, mode, gaps, band, literal, tb):
    """Long banded pairs (over 512 rows and 2^22 cells of the full matrix) in the lowest
    strips: heights at and around their edges, bands narrower and wider than a strip, a
    band whose strips start past the first column or hold no cell."""
    for m, n in [(2047, 2060), (2048, 2048), (2049, 2100), (2176, 2150), (2177, 2177), (4097, 1040), (1025, 4200)]:
        b = pairs(4, 900 + m, [(m, n)])
        q, r = b.pair(0)
        sc = dict(mode=mode, traceback=tb, band=band, band_literal=literal, **gaps)
        res, cig, rc = F.align_long(ctx, F.make_params(DNA_S, **sc), q, r)
        assert rc == 0, F.last_error()
        assert strip_rows(F, ctx) == 128
        o = oracle.align(q, r, DNA_S, **sc)
        fields = ("score", "q_end", "r_end", "status", "cells") + (("q_begin", "r_begin") if tb else ())
        for f in fields:
            assert int(res[f]) == int(o[f]), (m, n, f, int(res[f]), int(o[f]))
        if tb:
            assert np.array_equal(cig, o["cigar"]), (m, n)


@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("kind", ["local", "int32", "band"])
def test_waits_that_run_out(F, ctx, kind, tb):
    """Batches and captured pipelines whose pairs' first strips publish nothing, with a
    wait limit of 20 ms: every pair of the launch reports FILTR_ST_TIMEOUT, the calls
    that wait for the device report it too, and the context works on."""
    b = pairs(20, 15, [(600, 500), (200, 300), (1100, 900), (513, 64), (2000, 1500)])
    sc = dict(dict(affine=True, gap_open=11, gap_extend=1, traceback=tb), **KINDS[kind])
    params = F.make_params(b.subst, **sc)
    want = run(F, ctx, b, sc, 1)

    def timed_out(res):
        assert (res["status"] == 5).all()
        for f in ("score", "cells", "cigar_len"):
            assert (res[f] == 0).all(), f

    assert F.lib().filtr_test_set_strip_wait(ctx.handle, 1, 20_000_000) == F.OK
    F.lib().filtr_test_set_split(ctx.handle, 2)
    try:
        res, _, rc = F.align_batch(ctx, params, b)
        assert rc == F.OK
        timed_out(res)
        if tb:
            res, _, rc = F.align_batch(ctx, params, b, cigar_cap=10, raise_on_error=False)
            assert rc == F._lib.ERR_TIMEOUT
            timed_out(res)
        g = F.Graph(ctx, params, b.n, 2000, 1 << 30)
        try:
            res, _, status = F.graph_align(g, b)
            assert status == F._lib.ERR_TIMEOUT
            timed_out(res)
        finally:
            g.close()
    finally:
        F.lib().filtr_test_set_strip_wait(ctx.handle, 0, 0)
    same(run(F, ctx, b, sc, 2), want)
    g = F.Graph(ctx, params, b.n, 2000, 1 << 30)
    try:
        for _ in range(2):
            res, cig, status = F.graph_align(g, b)
            assert status == F.OK
            same((res, cig[:int(res["cigar_len"].sum())] if tb else want[1]), want)
    finally:
        g.close()


def test_tuned_contexts_keep_strips(F):
    """filtr_autotune, and its table applied elsewhere, leave the choice of a warp per
    strip to the batch's size; a table that prices the strips' shapes out does not."""
    b = pairs(20, 16, [(600, 500), (200, 300), (1100, 900), (513, 64), (2000, 1500)] * 6)
    sc = dict(mode="local", affine=True, gap_open=11, gap_extend=1, traceback=True)
    params = F.make_params(b.subst, **sc)
    c1, c2, c3 = F.Context(0, 4 << 30), F.Context(0, 1 << 30), F.Context(0, 1 << 30)
    try:
        table = c1.autotune(params)
        c2.tune_apply(params, table)
        forced = {f"{kind} R={r}": 1000.0 for kind, r in F.TUNE_SHAPES}
        forced["i16x2 R=24"] = 0.001
        c3.tune_apply(params, forced)
        want = None
        for c, strips in ((c1, True), (c2, True), (c3, False)):
            got = run(F, c, b, sc, 0)
            assert (strip_rows(F, c) > 0) == strips
            same(got, run(F, c, b, sc, 1))
            F.lib().filtr_test_set_split(c.handle, 0)
            # (every shape that a table may choose has strip buffers of up to 80 MB)
            g = F.Graph(c, params, b.n, 2000, 4 << 30)
            assert (strip_rows(F, c) > 0) == strips
            res, cig, status = F.graph_align(g, b)
            assert status == F.OK
            same((res, cig[:int(res["cigar_len"].sum())]), got)
            g.close()
            want = want or got
            same(got, want)
    finally:
        for c in (c1, c2, c3):
            c.close()


@pytest.mark.parametrize("kind,tb,n,length,strips", [
    ("local", True, 40, 1024, False), ("local", True, 40, 1025, True), ("local", False, 40, 1152, False),
    ("local", False, 40, 1153, True), ("band", True, 64, 300, True), ("band", False, 64, 512, False),
    ("band", False, 64, 513, True), ("local", False, 65, 1408, False), ("local", False, 255, 1409, True)])
def test_which_pipelines_take_strips(F, ctx, kind, tb, n, length, strips):
    F.lib().filtr_test_set_split(ctx.handle, 0)
    sc = dict(dict(affine=True, gap_open=11, gap_extend=1, traceback=tb), **KINDS[kind])
    g = F.Graph(ctx, F.make_params(PROT_S, **sc), n, length, 3 << 30)
    try:
        assert (strip_rows(F, ctx) > 0) == strips
    finally:
        g.close()
