"""The server's footprint estimate (CPU)."""
from paper_2511_16298_gb300 import serve


def test_default_estimate_refuses_no_more():
    """The default bound per request is not above the one it replaced."""
    for n in (1000, 1_000_000, 3_000_000):
        assert serve.estimate_bytes(n, 1920, 1080) <= 712 * n + 24 * 120 * 68
        assert serve.estimate_bytes(n, 4800, 64) <= 712 * n + 24 * 300 * 4
