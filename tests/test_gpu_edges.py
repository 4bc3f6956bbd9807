"""Decoder edges at chosen positions, and the larger grids, against the oracle."""
import numpy as np
import pytest

from paper_1312_0917_gb300 import binding as B
from gpu_util import assert_same_tracks, run_gpu
from test_gpu_stages import batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = B.Context(0)
    yield c
    c.close()


def road(hits, rng):
    """A road of `hits` hits (0 .. 40), dealt to the layers in turn: 3 + hits words."""
    w = [7 << 27 | int(rng.integers(0, 12)) | int(rng.integers(0, 6)) << 4 | int(rng.integers(0, 5)) << 7,
         5 << 27 | int(rng.integers(0, 1 << 16)), 6 << 27 | int(rng.integers(0, 1 << 16))]
    w += [(i % 5) << 27 | int(rng.integers(0, 4096)) for i in range(hits)]
    w[-1] |= 1 << 30
    return w


def stream(length, last, total, rng):
    """Roads whose ends include word `length` (the first `length` words are whole
    roads, the last of them of `last` words), then more up to `total` words."""
    roads, left = [], length - last
    while left:
        n = left if left in (3, 4, 5) else 3
        roads.append(road(n - 3, rng))
        left -= n
    roads.append(road(last - 3, rng))
    n, first = length, len(roads)
    while n < total:
        roads.append(road(40 if (len(roads) - first) % 200 == 0 else (10, 0, 11)[len(roads) % 3], rng))
        n += len(roads[-1])
    for i in range(len(roads)):
        if i % 200 == 199 or i + 1 == len(roads):
            roads[i][-1] |= 1 << 31
    return np.array([w for r in roads for w in r], np.uint32)


@pytest.mark.parametrize("edge,last", [(e, n) for e in (32, 64, 256, 1024, 2048) for n in (3, 13, 43) if n < e - 1])
def test_road_ends_around_an_edge(ctx, orc, consts, edge, last):
    """The last word of a road one before, at and one after the end of a window
    (32 words), of a group of windows (256) and of a decode step (1024, one CTA:
    spans of 2112 words), and a road of 43 words that starts there."""
    ctx.load_constants(consts, 1 << 40)
    for end in (edge - 1, edge, edge + 1):
        words = stream(end, last, 8 * 2100, np.random.default_rng(100 * edge + last))
        ends = np.nonzero((words >> 30) & 1)[0] + 1
        assert end in ends and (last == 3 or end - last == 0 or end - last in ends)
        rc, want = orc.run(words, consts, 1 << 40)
        assert rc == 0
        for max_ctas in (1, 0):
            ctx.set_launch(max_ctas=max_ctas)
            st, got, stats = run_gpu(ctx, words, B.PERSISTENT)
            ctx.set_launch()
            assert st == B.OK and stats["n_roads"] == len(ends)
            assert_same_tracks(got, want)


@pytest.mark.parametrize("events", [400, 560])
def test_larger_grids(ctx, orc, consts, cuts, events):
    """Two and three CTAs an SM by the words of the batch, against the oracle."""
    words = batch("grid", events, 64, 1, 4, seed=events)
    ctx.load_constants(consts, cuts["scaled"])
    st, got, _ = run_gpu(ctx, words, B.PERSISTENT)
    assert st == B.OK
    assert_same_tracks(got, orc.run(words, consts, cuts["scaled"])[1])
