"""The onesweep passes end whatever else the GPU runs: without the blocks that
make the tiles' prefixes (as if another stream held their SMs), and with two
sorts and two large frames at once on streams of their own."""
import threading

import numpy as np
import pytest
import torch

from paper_2511_16298_gb300 import synth
from paper_2511_16298_gb300 import tdgs as T

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2511_16298_gb300 import build
    build.build()


def pairs(m, bits, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    keys = torch.randint(0, 1 << bits, (m,), dtype=torch.int64, device=DEV, generator=g)
    return keys & ~(1 << 31), torch.arange(m, dtype=torch.int32, device=DEV)


# one tile, two, more tiles than blocks (several per block), the last ragged
@pytest.mark.parametrize("m,bits,flags", [(1, 44, 0), (4096, 44, 1), (4097, 44, 1), (300_001, 40, 0),
                                          (3_000_003, 45, 1)])
def test_without_prefix_blocks(m, bits, flags):
    keys, vals = pairs(m, bits, m)
    want, order = torch.sort(keys, stable=True)
    with T.Context(0) as ctx:
        for _ in range(2):
            k, v = ctx.diag_sort_pairs(keys.clone(), vals.clone(), bits - 32, flags)
            ctx.sync()
            assert torch.equal(k, want) and torch.equal(v.long(), order)
        k, v = ctx.sort_pairs(keys.clone(), vals.clone(), bits - 32, flags)
        ctx.sync()
        assert torch.equal(k, want) and torch.equal(v.long(), order)
        ctx.set_sort_variant(0)
        with pytest.raises(T.TdgsError) as e:
            ctx.diag_sort_pairs(keys.clone(), vals.clone(), bits - 32, flags)
        assert e.value.status == T.INVALID_ARGUMENT


def test_two_streams_at_once(oracle):
    """Each thread a context and a stream: sorts of 6M pairs on two, frames
    above one depth-sort launch on two."""
    frames = [synth.frame_random(i, 1_400_000 + i, 320, 200, max_sigma=3.0) for i in range(2)]
    refs = [oracle.sort_frame(f.gaussians, f.width, f.height) for f in frames]
    data = [pairs(6_000_000 + 5 * i, 44, i) for i in range(2)]
    sorted_ = [torch.sort(k, stable=True) for k, _ in data]
    recs = [T.records_to_tensor(f.gaussians, DEV) for f in frames]
    torch.cuda.synchronize()
    errors = []

    def sorts(i):
        for _ in range(8):
            k, v = ctx[i].sort_pairs(data[i][0].clone(), data[i][1].clone(), 12, T.SORT_DEPTH_POSITIVE)
            ctx[i].sync()
            assert torch.equal(k, sorted_[i][0]) and torch.equal(v.long(), sorted_[i][1])

    def views(i):
        for _ in range(8):
            k, v, r, m = ctx[2 + i].sort_frame(recs[i], frames[i].width, frames[i].height)
            ctx[2 + i].sync()
            assert m == refs[i]["m"]
        assert np.array_equal(k.cpu().numpy().view(np.uint64), refs[i]["keys"])
        assert np.array_equal(v.cpu().numpy().view(np.uint32), refs[i]["values"])

    def on_stream(fn, i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                fn(i)
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    ctx = [T.Context(0) for _ in range(4)]
    try:
        threads = [threading.Thread(target=on_stream, args=(fn, i)) for fn in (sorts, views) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors
    finally:
        for c in ctx:
            c.close()


@pytest.mark.parametrize("m", [(1 << 21) - 1, 1 << 21, (1 << 21) + 4097])
def test_histogram_with_one_and_four_steps(m):
    """Both sides of the size from which a histogram block takes four steps."""
    keys, vals = pairs(m, 44, m)
    want, order = torch.sort(keys, stable=True)
    with T.Context(0) as ctx:
        k, v = ctx.sort_pairs(keys, vals, 12)
        ctx.sync()
        assert torch.equal(k, want) and torch.equal(v.long(), order)
