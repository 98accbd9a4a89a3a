"""Decoders of few hidden units: padded to 8, 16, 32 or 64 inputs a layer and whole fours of outputs.
Against the 64-bit oracle at the library's bar for bfloat16 FNO outputs (2e-2 relative L2), and no
slower than a wide decoder's share of the work."""
import numpy as np
import pytest
import torch

import synth
from oracle import fno_oracle as fo

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import Fno, FnoShape  # noqa: E402


def _net(width, dec_layers, dec, cout, act):
    kw = dict(c_in=4, c_out=cout, width=width, layers=1, modes=4, dec_layers=dec_layers, dec_size=dec)
    s = synth.FnoShape(**kw)
    params = synth.fno_random_params(s, seed=2, out_scale=1.0)
    return Fno(FnoShape(**kw, activation=act), synth.fno_flatten_params(s, params)), s, params


@pytest.mark.parametrize("width,dec_layers,dec,cout,B,H,W,act", [
    (16, 1, 1, 16, 1, 16, 33, "gelu"), (16, 8, 4, 2, 2, 17, 40, "gelu"), (32, 2, 8, 9, 1, 16, 45, "relu"),
    (64, 3, 5, 1, 1, 16, 31, "gelu"), (16, 2, 9, 3, 1, 24, 40, "gelu"), (32, 8, 16, 16, 1, 16, 32, "gelu"),
    (64, 1, 12, 4, 2, 9, 33, "relu"), (48, 3, 17, 1, 1, 16, 40, "gelu"), (14, 2, 40, 2, 1, 16, 40, "gelu")])
def test_narrow_decoders_match_oracle(width, dec_layers, dec, cout, B, H, W, act):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    net, s, params = _net(width, dec_layers, dec, cout, 0 if act == "gelu" else 1)
    assert net.uses_tensor_cores(H, W)
    x = np.random.default_rng(4).standard_normal((B, 4, H, W)).astype(np.float32)
    y = net(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    net.check(B, H, W)
    want = fo.fno_forward(s, params, x, activation=act)
    assert np.linalg.norm(y - want) < 2e-2 * np.linalg.norm(want)


def test_narrow_decoders_take_less_time_than_wide_ones():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = torch.randn((8, 4, 256, 256), device="cuda")

    def ms(dec):
        net = _net(16, 8, dec, 1, 0)[0]
        y = torch.empty((8, 1, 256, 256), device="cuda")
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = float("inf")
        for _ in range(6):
            e[0].record()
            for _ in range(4):
                net(x, y)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        net.close()
        return best

    wide = ms(32)
    assert ms(16) < 0.8 * wide and ms(8) < 0.6 * wide and ms(1) < 0.6 * wide
