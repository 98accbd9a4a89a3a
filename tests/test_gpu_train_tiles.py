"""FNO training kernels at the edges of their tiles: widths that pad to 16, 32 and 64 channels,
rows around the pixel tiles, mode counts of every thread split of the x-DFT, wide and narrow
decoders, one to three outputs.  Against FP64 autograd; bar 2e-5 relative L2 per tensor (FP32
sums of at most some 10^4 terms, a root-of-n growth of the 6e-8 rounding, a few layers deep)."""
import numpy as np
import pytest
import torch

import synth
from oracle import grad_oracle as go

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import FnoShape  # noqa: E402
from paper_2604_27158_gb300.train import fno_apply  # noqa: E402

# width, modes, dec_layers, dec_size, c_in, c_out, B, H, W
CASES = [(2, 1, 1, 1, 1, 1, 1, 2, 2), (6, 5, 2, 7, 2, 1, 1, 11, 63), (14, 8, 1, 20, 1, 3, 2, 17, 65),
         (16, 13, 1, 16, 4, 2, 1, 26, 127), (18, 6, 1, 33, 4, 3, 3, 13, 129), (32, 12, 3, 32, 4, 3, 1, 25, 256),
         (34, 17, 1, 64, 3, 1, 1, 35, 257), (48, 20, 1, 48, 4, 3, 1, 65, 41), (64, 13, 1, 64, 4, 3, 1, 30, 200),
         (64, 32, 2, 64, 4, 3, 1, 64, 64), (20, 27, 1, 8, 16, 16, 1, 54, 55), (64, 30, 1, 3, 4, 3, 1, 61, 60)]


@pytest.mark.parametrize("width,modes,dec_layers,dec,cin,cout,B,H,W", CASES)
def test_training_kernels_at_tile_edges(width, modes, dec_layers, dec, cin, cout, B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=cin, c_out=cout, width=width, layers=2, modes=modes, dec_layers=dec_layers, dec_size=dec)
    s, g = synth.FnoShape(**kw), FnoShape(**kw)
    params = synth.fno_random_params(s, seed=5, out_scale=1.0)
    rng = np.random.default_rng(9)
    x = rng.standard_normal((B, cin, H, W)).astype(np.float32)
    dout = rng.standard_normal((B, cout, H, W)).astype(np.float32)
    pt = torch.from_numpy(synth.fno_flatten_params(s, params).astype(np.float32)).cuda().requires_grad_(True)
    xt = torch.from_numpy(x).cuda().requires_grad_(True)
    y = fno_apply(g, pt, xt)
    gp, gx = torch.autograd.grad(y, [pt, xt], torch.from_numpy(dout).cuda())
    p64 = go.bf16_params(params, requires_grad=True)
    x64 = torch.from_numpy(x.astype(np.float64)).requires_grad_(True)
    y64 = go.fno_forward(s, p64, x64, activation="gelu")
    (y64 * torch.from_numpy(dout.astype(np.float64))).sum().backward()

    def rel(a, b):
        return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))

    assert rel(y.detach().cpu().numpy().astype(np.float64), y64.detach().numpy()) < 2e-5
    assert rel(gx.cpu().numpy().astype(np.float64), x64.grad.numpy()) < 2e-5
    got, at = gp.cpu().numpy().astype(np.float64), 0
    scale = max(float(p64[name].grad.norm()) for name, _ in synth.fno_param_shapes(s))
    for name, shape in synth.fno_param_shapes(s):
        n = int(np.prod(shape))
        want = p64[name].grad.numpy().ravel()
        if np.linalg.norm(want) < 1e-15 * scale:  # identically zero (a sine at the Nyquist row): no direction
            assert np.linalg.norm(got[at:at + n]) < 2e-5 * scale, name
        else:
            assert rel(got[at:at + n], want) < 2e-5, name
        at += n
