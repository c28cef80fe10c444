"""Stored tuning tables (CPU): entries from before the interval splits, which
hold a tile digit width for every batch, are not applied; new ones round-trip,
and other entries stand."""
import json

import torch

from paper_2511_16298_gb300 import autotune


def test_entries_of_the_tile_passes_are_left_alone(tmp_path):
    views = [(torch.zeros((1000, 4), dtype=torch.int32), 1280, 720)]
    path = tmp_path / "tune.json"
    old = {"views:n10:t12:v1": {"knobs": {"tile_digit_bits": 8, "ctas_per_sm": 0, "depth_digit_bits": 0}, "ms": 1.0},
           "pairs:m10:tb12:f1": {"knobs": {"sort_variant": 2, "ctas_per_sm": 1}, "ms": 1.0}}
    path.write_text(json.dumps(old))
    table = autotune.Table(str(path))
    assert table.knobs_for_views(views) is None
    assert table.knobs_for_pairs(1000, 12, 1) == {"sort_variant": 2, "ctas_per_sm": 1}
    best = {"tile_digit_bits": 0, "ctas_per_sm": 2, "depth_digit_bits": 0}
    table.record({"key": autotune._views_key(views), "best": best, "ms": 0.5})
    table.save()
    again = autotune.Table(str(path))
    assert again.knobs_for_views(views) == best
    assert again.knobs_for_pairs(1000, 12, 1) == {"sort_variant": 2, "ctas_per_sm": 1}
