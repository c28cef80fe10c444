"""Reservations of asynchronous batches: what a refused batch or a failed
reservation leaves behind."""
import numpy as np
import pytest
import torch

from paper_2511_16298_gb300 import synth
from paper_2511_16298_gb300 import tdgs as T

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture
def ctx():
    from paper_2511_16298_gb300 import build
    build.build()
    c = T.Context(0)
    yield c
    c.close()


def on_gpu(frames):
    return [(T.records_to_tensor(f.gaussians, DEV), f.width, f.height) for f in frames]


def check(oracle, frames, results):
    assert len(frames) == len(results)
    for f, (k, v, r, m) in zip(frames, results):
        ref = oracle.sort_frame(f.gaussians, f.width, f.height)
        assert ref["status"] == 0 and m == ref["m"]
        assert np.array_equal(k.cpu().numpy().view(np.uint64), ref["keys"])
        assert np.array_equal(v.cpu().numpy().view(np.uint32), ref["values"])
        assert np.array_equal(r.cpu().numpy().view(np.uint32), ref["ranges"])


def refused(ctx, views):
    with pytest.raises(T.TdgsError) as e:
        ctx.sort_views_async(views)
    assert e.value.status == T.INVALID_ARGUMENT


def capture(ctx, views):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.sort_views_async(views)
    return graph


@pytest.mark.parametrize("n,size", [(3000, (640, 360)), (3000, (4800, 64))])
def test_refused_batches_stay_refused(ctx, oracle, n, size):
    """Batches of other counts (more Gaussians, more tiles, more views) are
    refused each time, and the reserved batch and its captured graph then give
    their own results: through the splits and the tile passes."""
    small = [synth.frame_random(i, n, *size) for i in range(2)]
    larger = [[synth.frame_random(5, n + 50_000, *size), small[1]],
              [small[0], synth.frame_random(6, n, size[0] * 2, size[1])], small + small[:1]]
    vs = on_gpu(small)
    cap = sum(oracle.sort_frame(f.gaussians, f.width, f.height)["m"] for f in small)
    ctx.reserve_views(vs, cap)
    ctx.sort_views_async(vs)
    graph = capture(ctx, vs)
    for frames in larger:
        vl = on_gpu(frames)
        refused(ctx, vl)
        refused(ctx, vl)
        graph.replay()
        check(oracle, small, ctx.views_results(2))
        ctx.sort_views_async(vs)
        check(oracle, small, ctx.views_results(2))


def test_failed_reservation_is_none(ctx, oracle):
    """A reservation for which there is no memory leaves none, not the one
    before with its buffers given up; arguments that are refused leave the one
    before."""
    frames = [synth.frame_random(1, 5000, 300, 200)]
    vs = on_gpu(frames)
    m = oracle.sort_frame(frames[0].gaussians, 300, 200)["m"]
    ctx.reserve_views(vs, m)
    with pytest.raises(T.TdgsError):
        ctx.reserve_views([(vs[0][0], 0, 200)], m)
    ctx.sort_views_async(vs)
    check(oracle, frames, ctx.views_results(1))
    torch.cuda.empty_cache()
    hold = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (24 << 30)), dtype=torch.uint8, device=DEV)
    with pytest.raises(T.TdgsError) as e:
        ctx.reserve_views(vs, 0xffffffff)
    assert e.value.status == T.OUT_OF_MEMORY
    refused(ctx, vs)
    del hold
    torch.cuda.empty_cache()
    ctx.reserve_views(vs, m)
    ctx.sort_views_async(vs)
    check(oracle, frames, ctx.views_results(1))


@pytest.mark.parametrize("dims,new", [([(320, 320), (320, 320)], [(6400, 16), (16, 6400)]),  # splits, then not
                                      ([(4800, 64), (4800, 64)], [(64, 4800), (4800, 64)])])  # tile passes both
def test_knobs_set_after_the_reservation(ctx, oracle, dims, new):
    """Batches keep the knobs of their reservation, which sized the scratch: a
    wider tile digit and more blocks set later wait for the next one."""
    first = [synth.frame_random(i, 20_000, w, h, max_sigma=5.0) for i, (w, h) in enumerate(dims)]
    other = [synth.frame_random(7 + i, 20_000, w, h, max_sigma=5.0) for i, (w, h) in enumerate(new)]
    vf, vo = on_gpu(first), on_gpu(other)
    cap = max(sum(oracle.sort_frame(f.gaussians, f.width, f.height)["m"] for f in x) for x in (first, other))
    ctx.apply_tuning({"tile_digit_bits": 0, "ctas_per_sm": 1})
    ctx.reserve_views(vf, cap)
    try:
        ctx.apply_tuning({"tile_digit_bits": 12, "ctas_per_sm": 8})
        for _ in range(2):
            ctx.sort_views_async(vo)
            check(oracle, other, ctx.views_results(2))
            ctx.sort_views_async(vf)
            check(oracle, first, ctx.views_results(2))
        ctx.reserve_views(vf, cap)
        ctx.sort_views_async(vo)
        check(oracle, other, ctx.views_results(2))
        check(oracle, first, ctx.sort_views(vf))
    finally:
        ctx.apply_tuning({"tile_digit_bits": 0, "ctas_per_sm": 0})


@pytest.mark.parametrize("width,height", [(640, 360), (4800, 64)])
@pytest.mark.parametrize("views", [1, 3])
def test_capacity_of_zero(ctx, width, height, views):
    """A reservation for no pairs takes batches without any, and reports the
    others, through the splits and the tile passes."""
    frames = [synth.frame_random(i, 2500, width, height) for i in range(views)]
    vs = on_gpu(frames)
    ctx.reserve_views(vs, 0)
    for _ in range(2):
        ctx.sort_views_async(vs)
        with pytest.raises(T.TdgsError) as e:  # (no result is read)
            ctx.views_results(views)
        assert e.value.status == T.CAPACITY
    for g, _, _ in vs:
        g[:, 3] = 0  # radius: culled
    ctx.sort_views_async(vs)
    graph = capture(ctx, vs)
    graph.replay()
    for k, v, r, m in ctx.views_results(views):
        assert m == 0 and k.numel() == 0 and not r.any()


@pytest.mark.parametrize("n", [3000, 700_000])  # the single-launch depth sort, and the passes with their scan
def test_captured_tile_passes_keep_their_scratch(ctx, oracle, n):
    """A captured batch through the tile passes outlives larger calls that
    take scratch of their own: normalised frames of both kinds, a scan and a
    sort by the chunked passes."""
    frames = [synth.frame_random(i, n, 4800, 64, max_sigma=5.0) for i in range(2)]
    vs = on_gpu(frames)
    ctx.reserve_views(vs, sum(oracle.sort_frame(f.gaussians, f.width, f.height)["m"] for f in frames))
    ctx.sort_views_async(vs)
    graph = capture(ctx, vs)
    for width, height in ((640, 360), (4800, 64)):
        f = synth.frame_random(9, 3 * n, width, height, max_sigma=5.0)
        st, ek, ev, er = oracle.sort_frame_normalized(f.gaussians, width, height)
        k, v, r, m = ctx.sort_frame_normalized(T.records_to_tensor(f.gaussians, DEV), width, height)
        assert st == 0 and m == len(ek)
        assert np.array_equal(k.cpu().numpy().view(np.uint32), ek)
        assert np.array_equal(v.cpu().numpy().view(np.uint32), ev)
    counts = torch.randint(0, 9, (9 * n,), dtype=torch.int32, device=DEV)
    off, _ = ctx.scan(counts)
    assert torch.equal(off[1:].long(), torch.cumsum(counts.long(), 0)[:-1])
    keys = torch.randint(0, 1 << 44, (9 * n,), dtype=torch.int64, device=DEV)
    vals = torch.arange(9 * n, dtype=torch.int32, device=DEV)
    want, order = torch.sort(keys, stable=True)
    ctx.set_sort_variant(0)
    sk, sv = ctx.sort_pairs(keys, vals, 12)
    ctx.set_sort_variant(-1)
    assert torch.equal(sk, want) and torch.equal(sv.long(), order)
    for _ in range(2):
        graph.replay()
        check(oracle, frames, ctx.views_results(2))


@pytest.mark.parametrize("shapes,new,fits", [
    ([(640, 160), (160, 640)], [(160, 640), (640, 160)], True),   # as many rows and columns at most
    ([(640, 160), (160, 640)], [(480, 160), (160, 800)], False),  # more rows in one view
    ([(320, 320), (320, 320)], [(640, 160), (160, 640)], False),  # wider and taller
    ([(1600, 64)], [(64, 1600)], False),
    ([(320, 320), (320, 320)], [(6400, 16), (16, 6400)], False),  # beyond the splits
])
def test_replays_of_other_proportions(ctx, oracle, shapes, new, fits):
    """A captured batch replayed over the table of a later one: its results
    where the captured launches have room for its rows and columns, and a
    report where they have not."""
    first = [synth.frame_random(i, 9000, w, h, max_sigma=5.0) for i, (w, h) in enumerate(shapes)]
    ns = [18_000] if len(new) == 1 else [7000, 11_000]
    other = [synth.frame_random(5 + i, k * len(shapes) // 2, w, h, max_sigma=5.0)
             for i, (k, (w, h)) in enumerate(zip(ns, new))]
    vf, vo = on_gpu(first), on_gpu(other)
    ctx.reserve_views(vf, max(sum(oracle.sort_frame(f.gaussians, f.width, f.height)["m"] for f in x)
                              for x in (first, other)))
    ctx.sort_views_async(vf)
    graph = capture(ctx, vf)
    ctx.sort_views_async(vo)
    check(oracle, other, ctx.views_results(len(vo)))
    graph.replay()
    if fits:
        check(oracle, other, ctx.views_results(len(vo)))
    else:
        with pytest.raises(T.TdgsError) as e:
            ctx.views_results(len(vo))
        assert e.value.status == T.CAPACITY
    ctx.sort_views_async(vf)
    check(oracle, first, ctx.views_results(len(vf)))


@pytest.mark.parametrize("n,width,height,sigma", [(4_000_000, 1280, 720, 0.5), (1_000_000, 1280, 720, 6.0),
                                                  (4_000_000, 4800, 1024, 0.5), (4_000_000, 4096, 4096, 0.5)])
def test_estimated_footprint(n, width, height, sigma):
    """The server's estimate bounds what a request holds, with few and with
    many pairs per Gaussian, and so does the documented size of a
    reservation."""
    from paper_2511_16298_gb300 import build, serve
    build.build()
    f = synth.frame_random(1, n, width, height, max_sigma=sigma)
    slack = 48 << 20  # allocations come in steps of 2 MB
    g = T.records_to_tensor(f.gaussians, DEV)
    with T.Context(0) as c:
        free = torch.cuda.mem_get_info()[0]
        m = c.sort_frame(g, width, height)[3]
        c.sync()
        used = free - torch.cuda.mem_get_info()[0]
        assert used + 16 * n <= serve.estimate_bytes(n, width, height, m / n) + slack, (used, m)
    with T.Context(0) as c:
        free = torch.cuda.mem_get_info()[0]
        c.reserve_views([(g, width, height)], m)
        used = free - torch.cuda.mem_get_info()[0]
        assert used <= 1.25 * (60 * n + 30 * m) + slack, (used, m)


@pytest.mark.parametrize("n,size", [(3000, (640, 360)), (3000, (4800, 64)), (700_000, (640, 360)),
                                    (700_000, (4800, 64))])
def test_first_call_is_a_capture(ctx, oracle, n, size):
    """A context whose first batch is captured and not yet replayed: what that
    batch clears is still to be cleared for the calls that run first (a batch
    outside the graph, or a frame of a second context)."""
    frames = [synth.frame_random(i, n, *size, max_sigma=5.0) for i in range(2)]
    vs = on_gpu(frames)
    cap = sum(oracle.sort_frame(f.gaussians, f.width, f.height)["m"] for f in frames)
    ctx.reserve_views(vs, cap)
    graph = capture(ctx, vs)
    ctx.sort_views_async(vs)
    check(oracle, frames, ctx.views_results(2))
    graph.replay()
    check(oracle, frames, ctx.views_results(2))
    with T.Context(0) as c:
        c.reserve_views(vs, cap)
        capture(c, vs)
        check(oracle, frames[:1], [c.sort_frame(*vs[0])])
        check(oracle, frames, c.sort_views(vs))
