"""Steps over 2^32 - 1 Gaussians, the most that a call takes: grids and
strides beyond it do not wrap (needs 105 GB)."""
import pytest
import torch

from paper_2511_16298_gb300 import synth
from paper_2511_16298_gb300 import tdgs as T

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_count_and_scan_of_the_most_gaussians():
    from paper_2511_16298_gb300 import build
    build.build()
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 110 << 30:
        pytest.skip("needs 105 GB of free device memory")
    n = 2 ** 32 - 1
    at = [0, 8191, 8192, 2 ** 31, n - 8192, n - 300, n - 1]  # visible ones, each with 4 pairs
    one = T.records_to_tensor(synth.records([16.0], [16.0], [1.0], [8]), DEV)
    with T.Context(0) as ctx:
        g = torch.zeros((n, 4), dtype=torch.int32, device=DEV)
        for i in at:
            g[i] = one[0]
        counts = ctx.count_tiles(g, 64, 64)
        ctx.sync()
        del g
        assert all(int(counts[i]) == 4 for i in at) and int(counts.sum(dtype=torch.int64)) == 4 * len(at)
        off, total = ctx.scan(counts)
        ctx.sync()
        assert int(total) == 4 * len(at)
        for k, i in enumerate(at):
            assert int(off[i]) == 4 * k
        assert int(off[n - 1]) == 4 * (len(at) - 1) and int(off[n - 2]) == 4 * (len(at) - 1)
    torch.cuda.empty_cache()
