"""A training pass of a narrow network does less work than that of a wider one on the same pixels,
so it takes no longer (10% for the spread of the timings): work that grows as layers get narrower,
such as a reduction over more partial sums, shows here."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import FnoShape  # noqa: E402
from paper_2604_27158_gb300.train import fno_apply  # noqa: E402


def _ms(width, B, H, W):
    kw = dict(c_in=4, c_out=1, width=width, layers=4, modes=8, dec_layers=1, dec_size=width)
    s = synth.FnoShape(**kw)
    params = synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)
    pt = torch.from_numpy(params).cuda().requires_grad_(True)
    x, dout = torch.randn((B, 4, H, W), device="cuda"), torch.randn((B, 1, H, W), device="cuda")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = float("inf")
    for _ in range(12):
        e[0].record()
        for _ in range(4):
            torch.autograd.grad(fno_apply(FnoShape(**kw), pt, x), [pt], dout)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("B,H,W", [(1, 486, 46), (8, 64, 64)])
def test_narrow_networks_train_no_slower_than_wide_ones(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wide = _ms(32, B, H, W)
    for width in (8, 16):
        assert _ms(width, B, H, W) < 1.1 * wide, width
