"""Rendering of records whose mean is not finite, in tiles with and without
the culling by the ellipse itself (more than 256 Gaussians).  A coordinate
that is no number blends everywhere, as in the oracle, which culls nothing; an
infinite one nowhere (the oracle's form of the exponent has inf - inf there:
it is given the same record far outside).  The bar of the render tests, with 15 of the
3072 pixels in place of one in a thousand for decisions that the exponentials'
last bits flip."""
import numpy as np
import pytest
import torch

from paper_2511_16298_gb300 import synth
from paper_2511_16298_gb300 import tdgs as T
from tests.test_gpu_render import BG, DEV, compare

pytestmark = pytest.mark.gpu
NAN, INF = np.nan, np.inf


@pytest.mark.parametrize("per_tile", [100, 400])
def test_means_that_are_not_finite(oracle, per_tile):
    from paper_2511_16298_gb300 import build
    build.build()
    W, H = 64, 48
    odd = [(NAN, 8.0), (8.0, NAN), (NAN, NAN), (NAN, 400.0), (-300.0, NAN), (INF, 20.0), (20.0, -INF), (INF, INF),
           (NAN, INF), (-INF, NAN), (8.0, 8.0), (NAN, 30.0)]
    rng = np.random.default_rng(per_tile)
    n = 12 * per_tile
    x, y = rng.uniform(-4, W + 4, n), rng.uniform(-4, H + 4, n)
    for t, (ox, oy) in enumerate(odd):
        x[t * per_tile + per_tile // 2], y[t * per_tile + per_tile // 2] = ox, oy
    rec = synth.records(x, y, np.full(n, 1.0), np.full(n, 9))
    s = rng.uniform(0.8, 3.0, (2, n))
    con = np.stack([1 / s[0] ** 2, rng.uniform(-0.5, 0.5, n) / (s[0] * s[1]), 1 / s[1] ** 2,
                    rng.uniform(0.02, 0.2, n)], 1).astype(np.float32)
    rgb = rng.random((n, 3)).astype(np.float32)
    values = np.arange(n, dtype=np.uint32)
    ranges = (np.arange(12)[:, None] * per_tile + np.array([0, per_tile])).astype(np.uint32)
    far = rec.copy()
    for c in ("x", "y"):
        far[c][np.isinf(rec["x"]) & ~np.isnan(rec["y"]) | np.isinf(rec["y"]) & ~np.isnan(rec["x"])] = 1e6
    st, want = oracle.render(far, con, rgb, values, ranges, W, H, BG)
    assert st == 0
    with T.Context(0) as ctx:
        img = ctx.render(T.records_to_tensor(rec, DEV), torch.from_numpy(con).to(DEV), torch.from_numpy(rgb).to(DEV),
                         torch.from_numpy(values.view(np.int32)).to(DEV),
                         torch.from_numpy(ranges.view(np.int32)).to(DEV), W, H, BG)
        ctx.sync()
        compare(img.cpu().numpy(), want, frac=5e-3)
