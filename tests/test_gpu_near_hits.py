"""Roads whose hits lie close together: many fits of a road then have the same
chi-square or nearly so.  The tracks equal the CPU oracle's bit for bit, and the
fit of such roads takes at most what deciding every one of them in whole keys
after the quick pass costs: one more pass of its own kind, not one road at a time."""
import numpy as np
import pytest

from paper_1312_0917_gb300 import binding as B
from gpu_util import torch_words
from test_gpu_stages import batch, check, p90

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


def test_ties_cost_one_more_pass(ctx, consts, cuts):
    """A tied road takes its warp step twice: with hits 16 strips apart the fit
    stage stays below three times its time with hits anywhere."""
    ctx.load_constants(consts, cuts["scaled"])
    words = batch("apart", 1000, 64, 1, 4)
    assert fit_us(ctx, near(words, 16)) < 3 * fit_us(ctx, words)


def test_repeats_cost_one_more_pass(ctx, consts, cuts):
    """The same for roads of which most hold a coordinate twice."""
    ctx.load_constants(consts, cuts["scaled"])
    words = batch("apart", 1000, 64, 1, 4)
    assert fit_us(ctx, near(words, 16, distinct=False)) < 3 * fit_us(ctx, words)
