"""The render kernel's culling of 8 x 4 pixel blocks, restated in float32
numpy and checked against the kernel's per-pixel cut test on extreme conics
(CPU; no GPU): with K = -2 cut, a block is left out when its columns lie
farther from the mean than sqrt(1.0201 K c / det) + 0.25, its rows farther
than sqrt(1.0201 K a / det) + 0.25, or (long tiles) the least d^T Q d over
the block grown by a quarter pixel exceeds 1.0201 K.  No left-out step may
pass the cut test, and the two tests together leave out at least as much as
the first alone."""
import numpy as np

from tests.test_render_cull_rule import f32, fma32, scene


def block_masks(x, y, con, tx0, ty0, ellipse):
    a, b, c, op = (con[:, k] for k in range(4))
    with np.errstate(all="ignore"):
        cut = np.where(op > 0, -np.log(f32(255.0) * op).astype(f32), f32(np.inf)).astype(f32)
        K = (f32(-2.0) * cut).astype(f32)
        ac = (a * c).astype(f32)
        det = fma32(-b, b, ac)
        ok = (a > 0) & (c > 0) & (det > f32(1e-3) * ac) & (K < f32(1e30))
        hy2 = ((K * a).astype(f32) / det).astype(f32) * f32(1.0201)
        hx2 = ((K * c).astype(f32) / det).astype(f32) * f32(1.0201)
        ok &= (hy2 < f32(1e30)) & (hx2 < f32(1e30))
        xr, yr = (x - tx0).astype(f32), (y - ty0).astype(f32)
        m = np.zeros(len(x), np.uint32)
        for w in range(8):
            c0, r0 = f32(8 * (w & 1)), f32(4 * (w >> 1))
            ex = np.maximum(np.maximum(c0 - xr, xr - (c0 + f32(7))) - f32(0.25), f32(0)).astype(f32)
            ey = np.maximum(np.maximum(r0 - yr, yr - (r0 + f32(3))) - f32(0.25), f32(0)).astype(f32)
            hit = ((ex * ex).astype(f32) <= hx2) & ((ey * ey).astype(f32) <= hy2)
            if ellipse:
                x0, y0 = (c0 - f32(0.25) - xr).astype(f32), (r0 - f32(0.25) - yr).astype(f32)
                x1, y1 = (x0 + f32(7.5)).astype(f32), (y0 + f32(3.5)).astype(f32)
                xe, ye = np.clip(f32(0), x0, x1), np.clip(f32(0), y0, y1)
                ys = np.clip(((-b / c).astype(f32) * xe).astype(f32), y0, y1)
                xs = np.clip(((-b / a).astype(f32) * ye).astype(f32), x0, x1)
                q1 = fma32(xe, fma32(a, xe, (f32(2) * b * ys).astype(f32)), (c * ys * ys).astype(f32))
                q2 = fma32(xs, fma32(a, xs, (f32(2) * b * ye).astype(f32)), (c * ye * ye).astype(f32))
                hit &= ~(np.minimum(q1, q2) > (K * f32(1.0201)).astype(f32))
            m |= hit.astype(np.uint32) << w
    return np.where(K < 0, 0, np.where(ok, m, 0xFF)).astype(np.uint32), cut


def test_block_culling_drops_only_steps_the_cut_test_drops():
    W, H = 320, 192
    x, y, rad, con = scene(12, 1500, W, H)
    t = np.arange(256)
    warp, lane = t >> 5, t & 31
    px, py = (warp & 1) * 8 + (lane & 7), (warp >> 1) * 4 + (lane >> 3)
    left = {False: 0, True: 0}
    total = 0
    for ty in range(H // 16):
        for tx in range(W // 16):
            tx0, ty0 = f32(tx * 16), f32(ty * 16)
            sel = (x + rad >= tx0) & (x - rad <= tx0 + 16) & (y + rad >= ty0) & (y - rad <= ty0 + 16)
            gx, gy, gc = x[sel], y[sel], con[sel]
            A, B, C = (f32(-0.5) * gc[:, 0]).astype(f32), (-gc[:, 1]).astype(f32), (f32(-0.5) * gc[:, 2]).astype(f32)
            dx = (gx[:, None] - (tx0 + px).astype(f32)[None, :]).astype(f32)
            dy = (gy[:, None] - (ty0 + py).astype(f32)[None, :]).astype(f32)
            for ellipse in (False, True):
                mask, cut = block_masks(gx, gy, gc, tx0, ty0, ellipse)
                with np.errstate(all="ignore"):
                    power = fma32(dx, fma32(A[:, None], dx, (B[:, None] * dy).astype(f32)),
                                  ((C[:, None] * dy).astype(f32) * dy).astype(f32))
                    passes = (power <= 0) & (power >= cut[:, None])
                kept = ((mask[:, None] >> warp[None, :]) & 1).astype(bool)
                assert not (passes & ~kept).any()
                left[ellipse] += int((~kept).sum())
            total += kept.size
    assert total > 1_000_000
    assert left[True] >= left[False] > 0.3 * total
