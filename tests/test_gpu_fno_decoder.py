"""Decoders the tensor-core decoder does not take -- several hidden layers, widths that are padded
to 32 or 64, more than three outputs, a last block that is not full -- against the FP64 oracle at
the library's bar for bfloat16 FNO outputs (2e-2 relative L2)."""
import numpy as np
import pytest
import torch

import synth
from oracle import fno_oracle as fo

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import Fno, FnoShape  # noqa: E402


@pytest.mark.parametrize("width,dec_layers,dec,cout,B,H,W,act", [
    (16, 3, 32, 1, 2, 24, 40, "gelu"), (16, 1, 7, 1, 1, 8, 64, "gelu"), (32, 2, 33, 3, 1, 17, 45, "gelu"),
    (32, 1, 32, 5, 1, 16, 32, "gelu"), (64, 3, 64, 2, 1, 16, 31, "gelu"), (14, 8, 64, 1, 1, 9, 33, "gelu"),
    (64, 2, 20, 16, 1, 16, 24, "relu"), (48, 2, 1, 1, 1, 16, 40, "relu")])
def test_deep_and_odd_decoders_match_oracle(width, dec_layers, dec, cout, B, H, W, act):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=4, c_out=cout, width=width, layers=1, modes=4, dec_layers=dec_layers, dec_size=dec)
    s = synth.FnoShape(**kw)
    params = synth.fno_random_params(s, seed=2, out_scale=1.0)
    net = Fno(FnoShape(**kw, activation=0 if act == "gelu" else 1), synth.fno_flatten_params(s, params))
    assert net.uses_tensor_cores(H, W)
    x = np.random.default_rng(4).standard_normal((B, 4, H, W)).astype(np.float32)
    y = net(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    net.check(B, H, W)
    want = fo.fno_forward(s, params, x, activation=act)
    assert np.linalg.norm(y - want) < 2e-2 * np.linalg.norm(want)
