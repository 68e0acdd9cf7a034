"""The persistent kernel and cluster size for several fp32 streams (host only):
one cluster serves one stream, and clusters beyond those resident at once run
in a second wave."""
import pytest

from paper_1905_00689_gb300 import FP32, plan

RESIDENT = {16: 7, 8: 15, 4: 36}


@pytest.mark.parametrize("H,K,B,variant,cluster", [
    (512, 64, 7, 1, 16), (512, 64, 8, 1, 8), (512, 64, 15, 1, 8), (512, 64, 16, 2, 4), (512, 64, 36, 2, 4),
    (512, 256, 8, 1, 16),                       # no smaller cluster holds it
    (256, 200, 7, 2, 16), (256, 200, 8, 1, 8),
    (200, 50, 15, 2, 8), (200, 50, 16, 2, 4),   # 48 terms per CTA or more: clusters of 8 up to one wave
    (256, 32, 1, 2, 4), (512, 16, 30, 2, 4),
])
def test_streams_choose_the_cluster(H, K, B, variant, cluster):
    p = plan(FP32, H, 20, B, K)
    assert (p["persistent_variant"], p["cluster"]) == (variant, cluster)
    if cluster < 16:
        assert B <= RESIDENT[cluster]


@pytest.mark.parametrize("H,K,B,variant,cluster", [
    (256, 128, 37, 2, 8), (256, 128, 46, 1, 4),   # three waves against two, four against two
    (256, 256, 8, 1, 8), (256, 256, 16, 2, 16), (256, 256, 22, 1, 8),
])
def test_many_terms_keep_the_one_exchange_kernel(H, K, B, variant, cluster):
    """The per-unit-block kernel on the smaller cluster takes 1.5 to 1.8 times as long."""
    p = plan(FP32, H, 20, B, K)
    assert (p["persistent_variant"], p["cluster"]) == (variant, cluster)
