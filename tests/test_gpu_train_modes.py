"""Spectral layers of few channels and many modes.  The y-transforms share their tables between the kx
of a warp, so a training pass of 8 channels takes a fraction of the time of 32 (a quarter of the
contractions; 0.6 leaves room for what does not shrink, and for the spread of the timings)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_2604_27158_gb300")
from train_timing import pass_ms  # noqa: E402


@pytest.mark.parametrize("B,H,W", [(32, 64, 58), (32, 500, 64)])
def test_narrow_spectral_layers_take_less_time_than_wide_ones(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wide = pass_ms(32, 29, 2, B, H, W)
    assert pass_ms(8, 29, 2, B, H, W) < 0.6 * wide


def test_few_rows_of_a_narrow_network_fill_the_chip():
    """The x-transform of 100 rows: blocks of whole warps of (row, channel) pairs would be seven for 8
    channels and 25 for 32, each as long (0.93 of the time in all then; 0.74 with a row a block)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert pass_ms(8, 29, 2, 1, 100, 1000) < 0.83 * pass_ms(32, 29, 2, 1, 100, 1000)
