"""A training pass of a narrow network does less work than that of a wider one on the same pixels,
so it takes no longer (10% for the spread of the timings): work that grows as layers get narrower,
such as a reduction over more partial sums, shows here."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_2604_27158_gb300")
from train_timing import pass_ms  # noqa: E402


@pytest.mark.parametrize("B,H,W", [(1, 486, 46), (8, 64, 64)])
def test_narrow_networks_train_no_slower_than_wide_ones(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wide = pass_ms(32, 8, 4, B, H, W)
    for width in (8, 16):
        assert pass_ms(width, 8, 4, B, H, W) < 1.1 * wide, width
