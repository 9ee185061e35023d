"""The integer multiply-add rate that bounds the fixed-point products: a warp's multiply-add holds its pipe for 4 to 5
FP32 FMA slots (29 lanes per clock and SM against 128), and three make one fixed-point multiply-add."""
import pytest

pytestmark = pytest.mark.gpu


def test_fixed_point_rate_is_a_share_of_the_fp32_peak(tgf):
    fixed = tgf.tgf_fma_peak(tgf.TGF_FMA_PEAK_FIXED)
    fp32 = tgf.tgf_fma_peak(tgf.TGF_FP32)
    assert 3 * 3.8 <= fp32 / fixed <= 3 * 5.2
