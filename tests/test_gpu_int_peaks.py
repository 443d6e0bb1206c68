"""The measured integer rates are roofs of the arithmetic that the kernels run: a split butterfly
(eight multiply instructions against ten) is the faster one, and large plain transforms stay below
the rate of their own butterfly, exact below N = 2^12 and split from there on."""
import os
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
K = pytest.importorskip("paper_2104_09583_gb300.copse")

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.fixture(scope="module")
def rates():
    ctx = K.copse_ctx_create(10, 55, 4, 2)
    try:
        return {kind: K.copse_measure_int_peak(ctx, kind, 5)[0] for kind in K.INT_PEAK_KINDS}
    finally:
        K.copse_ctx_destroy(ctx)


def test_split_butterflies_are_the_faster_ones(rates):
    # 10 / 8 = 1.25 where the multiplier alone bounds both; at least half of that
    assert rates["butterfly"] > 1.125 * rates["butterfly_exact"]
    # three multiply-adds against a butterfly's eight multiplies
    assert rates["mac"] > rates["butterfly"] > rates["barrett"]


@pytest.mark.parametrize("log_n", [11, 15])
@pytest.mark.parametrize("inverse", [False, True])
def test_transforms_stay_below_their_roof(rates, log_n, inverse):
    L = 16
    polys = (1 << 25) // (L << log_n)
    ctx = K.copse_ctx_create(log_n, 55, L, 3)
    try:
        x = torch.zeros(polys * L << log_n, dtype=torch.int64, device="cuda")
        family = "ntt_inv" if inverse else "ntt_fwd"
        for _ in range(3):
            K.copse_ntt(ctx, x.data_ptr(), polys, L, inverse=inverse)
        K.copse_stats_reset()
        K.copse_stats_enable(True)
        for _ in range(5):
            K.copse_ntt(ctx, x.data_ptr(), polys, L, inverse=inverse)
        torch.cuda.synchronize()
        K.copse_stats_enable(False)
        rate = K.copse_stats_get_ops(family) / (K.copse_stats_get(family)["ms"] * 1e-3)
        assert 0 < rate < rates[bench.peak_kind(family, log_n)]
    finally:
        K.copse_stats_enable(False)
        K.copse_stats_reset()
        K.copse_ctx_destroy(ctx)
