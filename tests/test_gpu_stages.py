"""The branches of the stages at the sizes where they change: fit classes and
their box fallback, the publishing of cross-road groups, the flag stage's rounds
and lists, the decoder's steps, the output's gathering, the grid by words and
the control block that each batch leaves empty.  All of it is integer work and
equals the CPU oracle bit for bit."""
import numpy as np
import pytest

from paper_1312_0917_gb300 import binding as B, synth
from gpu_util import assert_same_tracks, run_gpu, torch_words
from test_oracle_warrior import shared_cfg

pytestmark = pytest.mark.gpu
FLOAT_CUT = 1 << 24   # from this cut on the box path's float pass is used


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = B.Context(0, max_combinations=1 << 24)
    yield c
    c.close()


def batch(name, events, roads, lo, hi, shared=0.0, seed=1):
    return synth.make_batch(synth.Config(name, events, ("fixed", roads), ("uniform", lo, hi), shared_hits=shared),
                            seed=seed).words


def repeated(words):
    """The same stream with hit coordinates of two bits: repeats everywhere."""
    w = words.copy()
    hit = ((w >> 27) & 7) <= 4
    w[hit] = (w[hit] & np.uint32(0xFFFFF000)) | (w[hit] & np.uint32(3))
    return w


def p90(orc, words, consts):
    rc, chi = orc.chi2_all(words, consts)
    return int(np.sort(chi)[(9 * len(chi) + 9) // 10 - 1])


def check(ctx, orc, words, consts, cut, mode=B.PERSISTENT, **launch):
    ctx.load_constants(consts, cut)
    ctx.set_launch(**launch)
    try:
        st, got, stats = run_gpu(ctx, words, mode)
    finally:
        ctx.set_launch()
    rc, want = orc.run(words, consts, cut)
    assert st == B.OK and rc == 0
    assert_same_tracks(got, want)
    assert stats["n_passing"] == len(orc.run(words, consts, cut, warrior=-1)[1])
    return want, stats


# hits per layer: class by class, their edges (two and four hits in the smaller
# slots, four and eight in the larger), and what only the box path takes
SHAPES = [(1, 1), (1, 2), (2, 2), (1, 3), (2, 4), (3, 3), (4, 4), (1, 5), (2, 8), (4, 8), (5, 8), (8, 8)]


@pytest.mark.parametrize("kind", ["p90", "all", "ties", "small_cut", "repeats"])
@pytest.mark.parametrize("shape", SHAPES, ids=["%d-%d" % s for s in SHAPES])
def test_fit_classes(ctx, orc, consts, shape, kind):
    lo, hi = shape
    words = batch("shape", 3, 33 if hi <= 4 else 17, lo, hi, shared=0.3, seed=10 * lo + hi)
    if kind == "repeats":
        words = repeated(words)
    if kind in ("ties", "small_cut"):   # constants so small that many chi-squares are equal
        consts = {k: v.copy() for k, v in consts.items()}
        consts["C"] = (consts["C"] // 64).astype(np.int16)
        consts["k"] = consts["k"] * 0
    cut = {"all": 1 << 40, "small_cut": FLOAT_CUT - 1, "repeats": FLOAT_CUT}.get(kind)
    cut = p90(orc, words, consts) if cut is None else cut
    check(ctx, orc, words, consts, cut)
    check(ctx, orc, words, consts, cut, small_n4=16, run_roads=16)
    check(ctx, orc, words, consts, cut, mode=B.PLAIN)


@pytest.mark.parametrize("max_ctas", [0, 1])
@pytest.mark.parametrize("repeat", [False, True], ids=["distinct", "repeats"])
@pytest.mark.parametrize("lo,hi,roads", [(1, 3, 33), (1, 3, 160), (2, 4, 40), (3, 8, 20)])
def test_cross_road_groups(ctx, orc, consts, lo, hi, roads, repeat, max_ctas):
    """A word of candidates in many parts (all CTAs) and several words a warp
    (one CTA); candidates of the group path, of the box path and with repeated
    coordinates."""
    words = batch("groups", 4, roads, lo, hi, shared=0.7, seed=roads)
    words = repeated(words) if repeat else words
    cut = p90(orc, words, consts)
    _, a = check(ctx, orc, words, consts, cut, max_ctas=max_ctas)
    _, b = check(ctx, orc, words, consts, cut, mode=B.PLAIN)
    assert a["n_groups"] == b["n_groups"] and a["n_groups"] > 0


@pytest.mark.parametrize("block", [128, 256, 512])
@pytest.mark.parametrize("events", [5, 6, 7, 30])
def test_flag_stage_rounds_and_lists(ctx, orc, consts, events, block):
    """Two CTAs: up to three events each go to a CTA, more to a warp each
    (larger ones to a CTA); 30 events list more roads than a CTA gathers."""
    words = np.concatenate([batch("rounds", 1, (64, 33, 65, 200, 8)[i % 5], 1, 3, shared=0.5, seed=50 + i)
                            for i in range(events)])
    check(ctx, orc, words, consts, p90(orc, words, consts), block=block, max_ctas=2)


def diagonal_words(events, roads):
    """Roads of eight hits a layer, the same eight coordinates on every layer
    and no other road's."""
    words = batch("many", events, roads, 8, 8, seed=4)
    for layer in range(5):
        at = np.nonzero(((words >> 27) & 7) == layer)[0]
        words[at] = (words[at] & np.uint32(0xFFFFF000)) | (np.arange(len(at)) % (8 * roads)).astype(np.uint32)
    return words


@pytest.mark.parametrize("max_ctas", [0, 1, 3])
def test_output_beyond_what_a_cta_gathers(ctx, orc, consts, max_ctas):
    """Eight tracks a road (the chi-square is the sum of the squared differences
    of neighbouring layers), in one CTA and in many."""
    consts = {k: v * 0 for k, v in consts.items()}
    for r in range(3):
        consts["C"][:, r, r], consts["C"][:, r, r + 1] = 4096, -4096
    words = diagonal_words(5, 80)
    want, _ = check(ctx, orc, words, consts, 1 << 40, max_ctas=max_ctas)
    assert len(want) == 8 * 5 * 80


ROAD = np.array([7 << 27, 5 << 27, (6 << 27) | (1 << 30)], np.uint32)   # a road without hits


def end(words):
    w = words.copy()
    w[-1] |= np.uint32(1 << 31)
    return w


STREAMS = {
    "empty": np.zeros(0, np.uint32),
    "every word a header": np.full(3000, (7 << 27) | (1 << 30), np.uint32),
    "no header": np.full(5000, (1 << 27) | 5, np.uint32),
    "255 roads": end(np.tile(ROAD, 255)),
    "256 roads": end(np.tile(ROAD, 256)),
    "257 roads": end(np.tile(ROAD, 257)),
    "900 roads": end(np.tile(ROAD, 900)),
    "no end": np.tile(ROAD, 1000),
}


@pytest.mark.parametrize("max_ctas", [0, 1])
@pytest.mark.parametrize("name", STREAMS)
def test_decoder_at_the_limits(ctx, orc, consts, name, max_ctas):
    """Streams of nothing but one kind of word, more road starts in a step than
    are kept (384 in 1024 words), and roads per event around the limit; a good
    batch follows on the same context."""
    words = STREAMS[name]
    ctx.load_constants(consts, 1 << 40)
    for mode, launch in ((B.PERSISTENT, dict(max_ctas=max_ctas)), (B.PLAIN, {})):
        ctx.set_launch(**launch)
        st, got, _ = run_gpu(ctx, words, mode)
        rc, want = orc.run(words, consts, 1 << 40)
        assert st == rc
        if rc == 0:
            assert_same_tracks(got, want)
        check(ctx, orc, batch("after", 2, 20, 1, 3), consts, 1 << 40, mode=mode, **launch)


@pytest.mark.parametrize("cut_at", [31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 2047, 2048, 2049])
def test_decoder_at_the_edges_of_its_steps(ctx, orc, consts, cut_at):
    """Road ends around the edges of windows (32 words), groups of windows
    (256) and decode steps (1024): the stream's start is dropped word by word
    up to a road start, and one CTA takes long spans."""
    words = batch("edges", 240, 8, 0, 4, seed=cut_at)
    starts = np.nonzero((words >> 30) & 1)[0] + 1        # after a header
    first = int(starts[np.searchsorted(starts, len(words) - 8 * cut_at)])
    words = words[first:]
    rc, want = orc.run(words, consts, 1 << 40)
    ctx.load_constants(consts, 1 << 40)
    for max_ctas in (1, 2, 0):
        ctx.set_launch(max_ctas=max_ctas)
        st, got, _ = run_gpu(ctx, words, B.PERSISTENT)
        assert st == rc
        if rc == 0:
            assert_same_tracks(got, want)
    ctx.set_launch()


@pytest.mark.parametrize("events", [1, 90, 110, 400, 560])
def test_grid_by_words(ctx, orc, consts, cuts, events):
    """Batches on both sides of the lines at 640 and 3072 words an SM: the
    default grid gives the bytes of every grid."""
    words = batch("grid", events, 64, 1, 4, seed=events)
    ctx.load_constants(consts, cuts["scaled"])
    ctx.set_launch()
    st, ref, _ = run_gpu(ctx, words, B.PERSISTENT)
    assert st == B.OK
    if events <= 110:
        assert_same_tracks(ref, orc.run(words, consts, cuts["scaled"])[1])
    for bps in (1, 2, 3):
        ctx.set_launch(blocks_per_sm=bps)
        st, got, _ = run_gpu(ctx, words, B.PERSISTENT)
        assert st == B.OK and got.tobytes() == ref.tobytes()
    ctx.set_launch()


def test_control_block_is_left_empty(orc, consts):
    """Every way a batch can end leaves the control block empty for the next:
    unpacking alone, a fault, a limit, either mode; and a captured
    svt_fit_events replays between direct batches."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    good = batch("good", 6, 10, 1, 3, shared=0.6, seed=2)
    other = batch("other", 3, 12, 1, 4, seed=3)
    cut = p90(orc, good, consts)
    want, want_other = (orc.run(w, consts, cut)[1] for w in (good, other))
    c = B.Context(0, max_roads=256, max_combinations=1 << 20)
    c.load_constants(consts, cut)
    d = torch_words(good)
    try:
        for mode in (B.PERSISTENT, B.PLAIN):
            def good_batch():
                st, got, stats = run_gpu(c, good, mode, d_words=d)
                assert st == B.OK and stats["n_roads"] == 60
                assert_same_tracks(got, want)
            good_batch()
            assert c.unpack(d, len(good)) == B.OK
            for _ in range(2):
                assert len(c.get_roads()[1]) == 60
            good_batch()
            assert run_gpu(c, good[:-1], mode)[0] == orc.run(good[:-1], consts, cut)[0] != B.OK
            good_batch()
            assert run_gpu(c, np.concatenate([good] * 5), mode)[0] == B.E_CAPACITY
            good_batch()
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        assert c.unpack(d, len(good), s) == B.OK
        with torch.cuda.graph(g, stream=s):
            B.check(c.fit_events(B.PERSISTENT, s), "svt_fit_events")
        for _ in range(2):
            with torch.cuda.stream(s):
                g.replay()
            st, got = c.get_tracks(stream=s)
            assert st == B.OK
            assert_same_tracks(got, want)
            st, got, _ = run_gpu(c, other, B.PERSISTENT, stream=s)
            assert st == B.OK
            assert_same_tracks(got, want_other)
    finally:
        c.close()
