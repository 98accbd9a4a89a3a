"""Spectral layers of few channels and many modes: the y-transforms share their tables between the kx
of a warp, so a training pass of 8 channels takes a fraction of the time of 32 (a quarter of the
contractions; 0.6 leaves room for what does not shrink, and for the spread of the timings)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import FnoShape  # noqa: E402
from paper_2604_27158_gb300.train import fno_apply  # noqa: E402


def _ms(width, B, H, W):
    kw = dict(c_in=4, c_out=1, width=width, layers=2, modes=29, dec_layers=1, dec_size=width)
    s = synth.FnoShape(**kw)
    params = synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)
    pt = torch.from_numpy(params).cuda().requires_grad_(True)
    x, dout = torch.randn((B, 4, H, W), device="cuda"), torch.randn((B, 1, H, W), device="cuda")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = float("inf")
    for _ in range(8):
        e[0].record()
        for _ in range(4):
            torch.autograd.grad(fno_apply(FnoShape(**kw), pt, x), [pt], dout)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("B,H,W", [(32, 64, 58), (32, 500, 64)])
def test_narrow_spectral_layers_take_less_time_than_wide_ones(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wide = _ms(32, B, H, W)
    assert _ms(8, B, H, W) < 0.6 * wide


def test_few_rows_of_a_narrow_network_fill_the_chip():
    """The x-transform of 100 rows: blocks of whole warps of (row, channel) pairs would be seven for 8
    channels and 25 for 32, each as long (0.93 of the time in all then; 0.74 with a row a block)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert _ms(8, 1, 100, 1000) < 0.83 * _ms(32, 1, 100, 1000)
