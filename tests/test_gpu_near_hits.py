"""Roads whose hits lie close together: many fits of a road then have the same
chi-square or nearly so.  The tracks equal the CPU oracle's bit for bit, and the
fit of such roads takes at most what deciding every one of them in whole keys
after the quick pass costs: one more pass of its own kind, not one road at a time."""
import numpy as np
import pytest

from paper_1312_0917_gb300 import binding as B, synth
from gpu_util import torch_words
from test_gpu_stages import FLOAT_CUT, batch, check, p90

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = B.Context(0, max_combinations=1 << 24)
    yield c
    c.close()


def near(words, width, seed=1, distinct=True):
    """The same stream with a road's hits on a layer within `width` strips of
    one another (different strips, or drawn with repeats)."""
    rng = np.random.default_rng(seed)
    out = words.copy()
    kind = (out >> 27) & 7
    hit = kind <= 4
    road = np.cumsum(kind == 7) - 1
    row = (road[hit] * 5 + kind[hit]).astype(np.int64)
    order = np.argsort(row, kind="stable")
    new = np.r_[True, row[order][1:] != row[order][:-1]]
    at = np.arange(len(row))
    place = np.empty(len(row), np.int64)   # the hit's place in its layer
    place[order] = at - np.maximum.accumulate(np.where(new, at, 0))
    rows = 5 * (int(road[-1]) + 1)
    lo = rng.integers(0, 4096 - width + 1, size=rows)
    if distinct:
        off = np.argsort(rng.random((rows, width)), axis=1)[row, place]
    else:
        off = rng.integers(0, width, size=len(row))
    out[hit] = (out[hit] & np.uint32(0xFFFFF000)) | (lo[row] + off).astype(np.uint32)
    return out


def fit_us(c, words, reps=12):
    """Median time of the fit stage."""
    d = torch_words(words)
    t = []
    for _ in range(reps):
        assert c.unpack(d, len(words)) == B.OK
        assert c.fit_events(B.PERSISTENT) == B.OK
        t.append(c.get_stats()["phase_ns"][3] / 1e3)
    return float(np.median(t[3:]))


SMALL = [(1, 2), (2, 4), (1, 4), (3, 4), (1, 8)]


@pytest.mark.parametrize("width", [8, 64])
@pytest.mark.parametrize("lo,hi", SMALL, ids=["%d-%d" % s for s in SMALL])
def test_ties(ctx, orc, consts, lo, hi, width):
    words = near(batch("near", 4, 40, lo, hi, shared=0.2, seed=hi), width)
    cut = p90(orc, words, consts)
    check(ctx, orc, words, consts, cut)
    check(ctx, orc, words, consts, cut, mode=B.PLAIN)


@pytest.mark.parametrize("lo,hi", SMALL, ids=["%d-%d" % s for s in SMALL])
def test_repeated_coordinates(ctx, orc, consts, lo, hi):
    """Layers that hold a coordinate twice or more, fitted and excluded ones."""
    words = near(batch("near", 4, 40, lo, hi, shared=0.5, seed=hi), 8, distinct=False)
    cut = p90(orc, words, consts)
    _, a = check(ctx, orc, words, consts, cut)
    _, b = check(ctx, orc, words, consts, cut, mode=B.PLAIN)
    assert a["n_groups"] == b["n_groups"]


def test_every_fit_tied(ctx, orc, consts):
    """All chi-squares equal: the comb alone orders a road's fits."""
    flat = {k: v.copy() for k, v in consts.items()}
    flat["C"] = flat["C"] * 0
    for lo, hi in SMALL:
        words = batch("flat", 3, 30, lo, hi, seed=hi)
        check(ctx, orc, words, flat, 1 << 40)
        check(ctx, orc, words, flat, 1 << 40, mode=B.PLAIN)


BIG = [(5, 8), (4, 8), (8, 8)]


@pytest.mark.parametrize("width", [8, 16, 64])
@pytest.mark.parametrize("lo,hi", BIG, ids=["%d-%d" % s for s in BIG])
def test_near_candidates(ctx, orc, consts, lo, hi, width):
    """Roads of a warp each, with few and with many fits that floats cannot
    tell apart, above and below the cut from which floats are used."""
    words = near(batch("near", 2, 20, lo, hi, shared=0.2, seed=hi), width)
    cut = p90(orc, words, consts)
    check(ctx, orc, words, consts, cut)
    check(ctx, orc, words, consts, cut, mode=B.PLAIN)
    check(ctx, orc, words, consts, FLOAT_CUT)
    check(ctx, orc, words, consts, FLOAT_CUT - 1)
    check(ctx, orc, near(words, width, distinct=False), consts, cut)


def test_many_survivors(ctx, orc):
    """Roads of 8^4 fits of which those with c = a + b and e = a - b have
    chi-square zero, with a, b in 0..7, c in 0, 2, .. 14 and e in -6, -4, .. 8:
    one for each of the 32 pairs of like parity, no two with two hits in common,
    so that all of them survive."""
    from conftest import zero_consts
    flat = zero_consts()
    flat["C"][:, 0, :3] = 4096, 4096, -4096
    flat["C"][:, 1, :2], flat["C"][:, 1, 3] = (4096, -4096), -4096
    flat["k"][:, 0], flat["k"][:, 1] = 1000, 2000 + 6
    words = batch("many", 40, 1, 8, 8, seed=4)
    kind = (words >> 27) & 7
    road = np.cumsum(kind == 7) - 1
    excl = ((words >> 7) & 7)[kind == 7][road]
    for f, (first, step) in enumerate(((0, 1), (0, 1), (1000, 2), (2000, 2))):   # fitted layers in order
        for x in range(5):
            at = np.nonzero((excl == x) & (kind == f + (f >= x)))[0]
            words[at] = (words[at] & np.uint32(0xFFFFF000)) | (first + step * (np.arange(len(at)) % 8)).astype(np.uint32)
    want, _ = check(ctx, orc, words, flat, 1 << 40)
    assert len(want) >= 32 * 40
    check(ctx, orc, words, flat, 1)
    check(ctx, orc, words, flat, 1 << 40, mode=B.PLAIN)


def test_ties_cost_one_more_pass(ctx, consts, cuts):
    """A tied road takes its warp step twice: with hits 16 strips apart the fit
    stage stays below three times its time with hits anywhere."""
    ctx.load_constants(consts, cuts["scaled"])
    words = batch("apart", 1000, 64, 1, 4)
    assert fit_us(ctx, near(words, 16)) < 3 * fit_us(ctx, words)


def test_tied_steps_are_evened_out(ctx, consts, cuts):
    """Roads of skewed hit counts, four steps a warp, some of them taken twice: the
    fit stays below twice its time with hits anywhere."""
    ctx.load_constants(consts, cuts["uneven"])
    words = synth.make_batch(synth.Config("skew", 3000, ("geom", 32, 1, 256), ("skewed", 8)), seed=1).words
    assert fit_us(ctx, near(words, 16)) < 2 * fit_us(ctx, words)


def test_repeats_cost_one_more_pass(ctx, consts, cuts):
    """The same for roads of which most hold a coordinate twice."""
    ctx.load_constants(consts, cuts["scaled"])
    words = batch("apart", 1000, 64, 1, 4)
    assert fit_us(ctx, near(words, 16, distinct=False)) < 3 * fit_us(ctx, words)


@pytest.mark.parametrize("kind", ["near", "small_cut"])
def test_near_candidates_cost_one_pass(ctx, consts, cuts, kind):
    """Whole keys for every fit take less than twice the pass in floats."""
    words = batch("apart", 100, 128, 8, 8)
    ctx.load_constants(consts, cuts["stress"])
    t = fit_us(ctx, words)
    if kind == "small_cut":
        ctx.load_constants(consts, FLOAT_CUT - 1)
    assert fit_us(ctx, near(words, 16) if kind == "near" else words) < 2 * t
