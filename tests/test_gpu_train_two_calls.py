"""Training passes of one shape whose backward runs later: every call keeps its own activations."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import FnoShape  # noqa: E402
from paper_2604_27158_gb300.train import fno_apply  # noqa: E402


@pytest.mark.parametrize("act", [0, 1])
def test_two_forwards_before_their_backwards(act):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=4, c_out=3, width=16, layers=2, modes=4, dec_layers=1, dec_size=32)
    s, g = synth.FnoShape(**kw), FnoShape(**kw, activation=act)
    p = torch.from_numpy(synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)).cuda()
    p.requires_grad_(True)
    gen = torch.Generator(device="cuda").manual_seed(3)
    xs = [torch.randn((2, 4, 24, 40), generator=gen, device="cuda").requires_grad_(True) for _ in range(2)]
    dout = torch.randn((2, 3, 24, 40), generator=gen, device="cuda")
    want = [torch.autograd.grad(fno_apply(g, p, x), [p, x], dout) for x in xs]
    ys = [fno_apply(g, p, x) for x in xs]
    got = [torch.autograd.grad(y, [p, x], dout) for y, x in zip(ys, xs)]
    for a, b in zip(got, want):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    (gp,) = torch.autograd.grad(sum((fno_apply(g, p, x) * dout).sum() for x in xs), [p])
    torch.testing.assert_close(gp, want[0][0] + want[1][0], rtol=1e-6, atol=0)


def test_activations_are_given_back_after_the_backward():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=4, c_out=3, width=32, layers=4, modes=12, dec_layers=1, dec_size=32)
    s, g = synth.FnoShape(**kw), FnoShape(**kw)
    p = torch.from_numpy(synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)).cuda()
    p.requires_grad_(True)
    x = torch.randn((2, 4, 64, 128), device="cuda")
    losses = []
    for k in range(4):
        losses.append((fno_apply(g, p, x) ** 2).mean())  # kept, with its graph
        losses[-1].backward()
        torch.cuda.synchronize()
        if k == 0:
            held = torch.cuda.memory_allocated()
    assert torch.cuda.memory_allocated() <= held + (8 << 20)
