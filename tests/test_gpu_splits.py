"""Frames whose pairs come from the interval splits (rows, then columns), at
the sizes where the launches change form: 32-item batches, 1024-item tiles,
tile rows and columns per 32-bit word, tiles with more pairs than are staged
at once, the depth sort's tile sizes and the image size above which the tile
passes take over.  Every output equals the CPU oracle's bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_16298_gb300 import synth
from paper_2511_16298_gb300 import tdgs as T

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    from paper_2511_16298_gb300 import build
    build.build()
    c = T.Context(0)
    yield c
    c.close()


def same(ctx, oracle, fr):
    ref = oracle.sort_frame(fr.gaussians, fr.width, fr.height)
    assert ref["status"] == 0
    k, v, r, m = ctx.sort_frame(T.records_to_tensor(fr.gaussians, DEV), fr.width, fr.height)
    ctx.sync()
    assert m == ref["m"]
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["keys"])
    assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["values"])
    assert np.array_equal(r.cpu().numpy().view(np.uint32), ref["ranges"])


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 2048, 2049, 4097, 32_768, 32_769, 70_001])
def test_item_counts(ctx, oracle, n):
    same(ctx, oracle, synth.frame_random(n, n, 333, 209, depth_ties=0.3))


@pytest.mark.parametrize("n", [5000, 33_000])
@pytest.mark.parametrize("cols,rows", [(1, 1), (1, 70), (32, 33), (33, 32), (64, 65), (65, 64), (96, 97), (97, 96),
                                       (160, 161), (161, 160), (224, 225), (225, 224), (256, 3), (3, 256),
                                       (256, 256), (257, 2), (2, 257)])
def test_grid_sizes(ctx, oracle, cols, rows, n):
    """Rows and columns on both sides of each compiled width, 256 (the most
    that the splits take) and 257, for the one-launch form of small frames and
    the launch per step."""
    same(ctx, oracle, synth.frame_random(cols * 1000 + rows, n, 16 * cols - 7, 16 * rows - 3, max_sigma=90.0))


def covering(n, width, height, seed, small=0.0):
    """Gaussians over the whole image (a share of them a few pixels wide)."""
    rng = np.random.default_rng(seed)
    r = np.full(n, 4 * max(width, height))
    r[rng.random(n) < small] = 5
    return synth.Frame(width, height, synth.records(rng.uniform(0, width, n), rng.uniform(0, height, n),
                                                    rng.uniform(0.5, 4.0, n).round(1), r), "covering")


@pytest.mark.parametrize("n,width,height,small", [(1100, 4096, 48, 0.0), (1500, 640, 360, 0.5), (1030, 16, 16, 0.0),
                                                  (700, 48, 4096, 0.3)])
def test_windows_of_bins(ctx, oracle, n, width, height, small):
    """Tiles with several times the pairs that are staged at once: windows
    of whole rows or columns, in which some items have no bins."""
    same(ctx, oracle, covering(n, width, height, n, small))


@pytest.mark.parametrize("width,height", [(4096, 48), (640, 360), (48, 4096)])
def test_windows_of_bins_among_many(ctx, oracle, width, height):
    """The same above the one-launch form: 1100 covering Gaussians in front of
    34,000 small ones, so that whole tiles are covering."""
    rng = np.random.default_rng(width)
    front = covering(1100, width, height, 5)
    front.gaussians["depth"] = rng.uniform(0.3, 0.4, 1100).astype(np.float32)
    rest = synth.frame_random(6, 34_000, width, height, max_sigma=3.0)
    rest.gaussians["depth"] += 1.0
    g = np.concatenate([rest.gaussians, front.gaussians])[rng.permutation(35_100)]
    same(ctx, oracle, synth.Frame(width, height, g, "front"))


@pytest.mark.parametrize("per_sm", [2048, 4096])
def test_depth_sort_tile_sizes(ctx, oracle, per_sm):
    """Frames that just fill, and just overflow, one depth-sort tile of 4 or 8
    keys per thread on every SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (sms * per_sm, sms * per_sm + 1):
        same(ctx, oracle, synth.frame_scene(n, n=n, width=640, height=360))


def test_no_pairs_and_culled(ctx, oracle):
    fr = synth.frame_random(3, 3000, 500, 300)
    fr.gaussians["radius"] = 0
    same(ctx, oracle, fr)
    fr.gaussians["radius"][1234] = 9
    same(ctx, oracle, fr)


def test_async_one_view_capacity_then_exact(ctx, oracle):
    """One reserved view: more pairs than the capacity are reported and leave
    the context usable; within it, a tile digit width set after the
    reservation does not change the reserved path."""
    fr = synth.frame_small(2)
    ref = oracle.sort_frame(fr.gaussians, fr.width, fr.height)
    g = T.records_to_tensor(fr.gaussians, DEV)
    views = [(g, fr.width, fr.height)]
    ctx.reserve_views(views, ref["m"] - 1)
    ctx.sort_views_async(views)
    with pytest.raises(T.TdgsError) as e:
        ctx.views_results(1)
    assert e.value.status == T.CAPACITY
    ctx.reserve_views(views, ref["m"])
    ctx.apply_tuning({"tile_digit_bits": 8})
    try:
        for _ in range(2):
            ctx.sort_views_async(views)
            (k, v, r, m), = ctx.views_results(1)
            assert m == ref["m"]
            assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["keys"])
            assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["values"])
            assert np.array_equal(r.cpu().numpy().view(np.uint32), ref["ranges"])
    finally:
        ctx.apply_tuning({"tile_digit_bits": 0})
    same(ctx, oracle, fr)


def depths(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "equal":
        return np.full(n, 2.5)
    if kind == "narrow":
        return rng.uniform(1.0, 1.0001, n)
    return np.exp(rng.uniform(np.log(1e-37), np.log(1e37), n))


@pytest.mark.parametrize("kind", ["equal", "narrow", "wide"])
@pytest.mark.parametrize("sizes", [(700, 0, 1, 2500), (1030, 5000, 40_000), (650_000, 3, 700_000)])
def test_batches_in_view_order(ctx, oracle, kind, sizes):
    """Batches whose depth keys need one to four digit passes, then the pass
    by view: the single launch at two tile sizes and the onesweep passes,
    with empty and tiny views among the others."""
    frames = []
    for i, n in enumerate(sizes):
        f = synth.frame_random(40 + i, n, 300 + 50 * i, 200, max_sigma=8.0) if n else synth.Frame(
            64, 64, synth.records([], [], [], []), "empty")
        if n:
            f.gaussians["depth"] = depths(kind, n, i).astype(np.float32)
        frames.append(f)
    res = ctx.sort_views([(T.records_to_tensor(f.gaussians, DEV), f.width, f.height) for f in frames])
    for f, (k, v, r, m) in zip(frames, res):
        ref = oracle.sort_frame(f.gaussians, f.width, f.height)
        assert ref["status"] == 0 and m == ref["m"]
        assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["keys"])
        assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["values"])
        assert np.array_equal(r.cpu().numpy().view(np.uint32), ref["ranges"])


@pytest.mark.parametrize("n,width,height", [(1, 16, 16), (2049, 4096, 50), (2049, 4112, 50), (50_000, 700, 500),
                                            (1_300_000, 320, 200)])
def test_normalized_key(ctx, oracle, n, width, height):
    """The 32-bit normalised key through the splits (the single-launch and the
    onesweep depth sort) and, above 4096 pixels, through the five steps."""
    fr = synth.frame_random(n % 97, n, width, height, max_sigma=6.0 if n > 100_000 else 64.0, depth_ties=0.2)
    st, ek, ev, er = oracle.sort_frame_normalized(fr.gaussians, width, height)
    assert st == 0
    k, v, r, m = ctx.sort_frame_normalized(T.records_to_tensor(fr.gaussians, DEV), width, height)
    ctx.sync()
    assert m == len(ek)
    assert np.array_equal(k.cpu().numpy().view(np.uint32), ek)
    assert np.array_equal(v.cpu().numpy().view(np.uint32), ev)
    assert np.array_equal(r.cpu().numpy().view(np.uint32), er)


@pytest.mark.parametrize("n,cap", [(1, None), (33, None), (5000, None), (5000, 1), (5000, 0.5), (70_001, None)])
def test_duplicate_and_ranges_steps(ctx, oracle, n, cap):
    """duplicate_keys with runs of culled Gaussians and whole-screen ones, with
    and without room for every pair, and tile_ranges at sizes around a warp's
    128 keys: the pairs written are the oracle's, and the missing ones are
    reported."""
    fr = synth.frame_random(n, n, 777, 331, max_sigma=200.0, culled=0.4)
    ref = oracle.sort_frame(fr.gaussians, fr.width, fr.height)
    m = ref["m"]
    g = T.records_to_tensor(fr.gaussians, DEV)
    off = torch.from_numpy(ref["offsets"].view(np.int32)).to(DEV)
    room = m if cap is None else (cap if cap >= 1 else int(m * cap))
    k, v = ctx.duplicate_keys(g, off, fr.width, fr.height, room)
    if room < m:
        with pytest.raises(T.TdgsError) as e:
            ctx.sync()
        assert e.value.status == T.CAPACITY
    else:
        ctx.sync()
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["unsorted_keys"][:room])
    assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["unsorted_values"][:room])
    sk = torch.from_numpy(ref["keys"].view(np.int64)).to(DEV)
    for mm in sorted({min(x, m) for x in (1, 31, 32, 33, 127, 128, 129, 1024, 1025, m)}):
        r = ctx.tile_ranges(sk, fr.num_tiles, m=mm)
        ctx.sync()
        tiles = (ref["keys"][:mm] >> np.uint64(32)).astype(np.int64)
        want = np.zeros((fr.num_tiles, 2), np.uint32)
        want[:, 0] = np.searchsorted(tiles, np.arange(fr.num_tiles), "left")
        want[:, 1] = np.searchsorted(tiles, np.arange(fr.num_tiles), "right")
        want[want[:, 0] == want[:, 1]] = 0
        assert np.array_equal(r.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("n", [5000, 60_000])
def test_normalized_key_first_call(oracle, n):
    """A context's first call: nothing is allocated yet."""
    fr = synth.frame_random(n, n, 500, 300)
    st, ek, ev, er = oracle.sort_frame_normalized(fr.gaussians, fr.width, fr.height)
    assert st == 0
    c = T.Context(0)
    try:
        k, v, r, m = c.sort_frame_normalized(T.records_to_tensor(fr.gaussians, DEV), fr.width, fr.height)
        c.sync()
        assert m == len(ek)
        assert np.array_equal(k.cpu().numpy().view(np.uint32), ek)
        assert np.array_equal(v.cpu().numpy().view(np.uint32), ev)
        assert np.array_equal(r.cpu().numpy().view(np.uint32), er)
    finally:
        c.close()


def test_normalized_call_keeps_frames(ctx, oracle):
    """A frame's results, a batch between its asynchronous call and its
    results, and a captured batch all outlive a larger normalised-key frame on
    the same context."""
    a, b = synth.frame_random(1, 3000, 320, 200), synth.frame_random(2, 60_000, 1000, 700)
    ga, gb = T.records_to_tensor(a.gaussians, DEV), T.records_to_tensor(b.gaussians, DEV)
    ref = oracle.sort_frame(a.gaussians, a.width, a.height)

    def equal(res):
        assert res[3] == ref["m"]
        assert np.array_equal(res[0].cpu().numpy().view(np.uint64), ref["keys"])
        assert np.array_equal(res[1].cpu().numpy().view(np.uint32), ref["values"])
        assert np.array_equal(res[2].cpu().numpy().view(np.uint32), ref["ranges"])

    c = T.Context(0)
    try:
        res = c.sort_frame(ga, a.width, a.height)
        c.sort_frame_normalized(gb, b.width, b.height)
        equal(res)
        views = [(ga, a.width, a.height)] * 2
        c.reserve_views(views, 2 * ref["m"])
        c.sort_frame_normalized(gb, b.width, b.height)
        c.sort_views_async(views)  # (the reservation still stands)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            c.sort_views_async(views)
        k, v, r, m = c.sort_frame_normalized(gb, b.width, b.height)
        for x in c.views_results(2):
            equal(x)
        graph.replay()
        for x in c.views_results(2):
            equal(x)
        st, ek, ev, er = oracle.sort_frame_normalized(b.gaussians, b.width, b.height)
        assert st == 0 and m == len(ek)
        assert np.array_equal(k.cpu().numpy().view(np.uint32), ek)
        assert np.array_equal(v.cpu().numpy().view(np.uint32), ev)
        assert np.array_equal(r.cpu().numpy().view(np.uint32), er)
    finally:
        c.close()


@pytest.mark.parametrize("n,shapes,new", [
    (20_000, [(1600, 64)], [(64, 1600)]),                              # one view, turned
    (20_000, [(640, 160), (160, 640)], [(160, 640), (640, 160)]),      # two views exchanged
    (20_000, [(320, 320), (320, 320)], [(6400, 16), (16, 6400)]),      # beyond the splits' 256 columns and rows
    (700_000, [(320, 320), (320, 320)], [(640, 160), (160, 640)]),     # above one depth-sort launch
])
def test_reservation_takes_other_proportions(ctx, oracle, n, shapes, new):
    """A reservation is for counts of views, Gaussians and tiles: batches with
    the same totals in other proportions, and views with other Gaussian
    counts, give their own results through the asynchronous call; replays of
    the captured batch read the table staged last, and give its results or
    report that they have no room for them."""
    def batch(dims, split, seed):
        ns = [n] if len(dims) == 1 else [int(n * split), 2 * n - int(n * split)]
        return [synth.frame_random(seed + i, k, w, h, max_sigma=5.0) for i, (k, (w, h)) in enumerate(zip(ns, dims))]

    def on_gpu(frames):
        return [(T.records_to_tensor(f.gaussians, DEV), f.width, f.height) for f in frames]

    def check(frames, res):
        for f, (k, v, r, m) in zip(frames, res):
            ref = oracle.sort_frame(f.gaussians, f.width, f.height)
            assert ref["status"] == 0 and m == ref["m"]
            assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["keys"])
            assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["values"])
            assert np.array_equal(r.cpu().numpy().view(np.uint32), ref["ranges"])

    first, other = batch(shapes, 1.0, 1), batch(new, 0.31, 7)
    vf, vo = on_gpu(first), on_gpu(other)
    c = T.Context(0)
    try:
        cap = max(sum(x[3] for x in c.sort_views(v)) for v in (vf, vo)) + 100
        c2 = T.Context(0)  # sized by the reservation alone
        try:
            c2.reserve_views(vf, cap)
            c2.sort_views_async(vf)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                c2.sort_views_async(vf)
            check(first, c2.views_results(len(vf)))
            c2.sort_views_async(vo)
            check(other, c2.views_results(len(vo)))
            graph.replay()  # (reads the table of `other`)
            try:
                check(other, c2.views_results(len(vo)))
            except T.TdgsError as e:
                assert e.status == T.CAPACITY and new != shapes
            c2.sort_views_async(vf)
            check(first, c2.views_results(len(vf)))
        finally:
            c2.close()
    finally:
        c.close()
