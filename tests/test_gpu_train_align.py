"""Training calls whose saved activations lie at an address that is 8-byte but not 16-byte aligned:
the same bits as with an aligned buffer (only the width of loads and stores may differ)."""
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300._abi import call  # noqa: E402
from paper_2604_27158_gb300.fno import FnoShape  # noqa: E402
from paper_2604_27158_gb300.train import fno_train_query  # noqa: E402

# width, modes, dec_layers, dec_size, c_in, c_out, B, H, W: every tile shape of the pointwise kernel,
# widths of whole and of broken 16-byte units
CASES = [(8, 4, 1, 16, 2, 1, 2, 17, 33), (16, 5, 3, 32, 4, 4, 1, 20, 129), (64, 13, 1, 64, 4, 3, 1, 30, 200),
         (32, 12, 2, 24, 2, 2, 2, 25, 256), (6, 3, 1, 7, 1, 1, 1, 11, 15)]


@pytest.mark.parametrize("act", [0, 1])
@pytest.mark.parametrize("width,modes,dec_layers,dec,cin,cout,B,H,W", CASES)
def test_saved_activations_at_eight_byte_addresses(act, width, modes, dec_layers, dec, cin, cout, B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=cin, c_out=cout, width=width, layers=2, modes=modes, dec_layers=dec_layers, dec_size=dec)
    s = synth.FnoShape(**kw)
    g = FnoShape(**kw, activation=act)
    params = torch.from_numpy(synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((B, cin, H, W), generator=gen, device="cuda")
    dout = torch.randn((B, cout, H, W), generator=gen, device="cuda")
    sz, cfg = fno_train_query(g, B, H, W), g.c()
    ws = torch.empty(sz.ws_bytes + 256, dtype=torch.uint8, device="cuda")
    wp = ws.data_ptr() + (-ws.data_ptr()) % 256
    buf = torch.empty(sz.saved_bytes // 4 + 8, device="cuda")
    got = []
    for off in (0, 2):  # floats
        saved = buf.data_ptr() + (-buf.data_ptr()) % 16 + 4 * off
        out, dp, dx = torch.empty_like(dout), torch.empty_like(params), torch.empty_like(x)
        call("fno_train_forward", ctypes.byref(cfg), params.data_ptr(), x.data_ptr(), out.data_ptr(), B, H, W, saved,
             wp, None)
        call("fno_train_backward", ctypes.byref(cfg), params.data_ptr(), dout.data_ptr(), saved, dp.data_ptr(),
             dx.data_ptr(), B, H, W, wp, None)
        torch.cuda.synchronize()
        got.append((out, dp, dx))
    for a, b in zip(*got):
        assert torch.equal(a, b)
