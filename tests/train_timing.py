"""Device time of a training pass (forward and backward, by the C ABI), without the host's."""
import ctypes

import numpy as np
import torch

import synth


def pass_ms(width, modes, layers, B, H, W):
    """Milliseconds of one pass, best of ten replays of a captured graph of four."""
    from paper_2604_27158_gb300._abi import call
    from paper_2604_27158_gb300.fno import FnoShape
    from paper_2604_27158_gb300.lbm import _stream_ptr
    from paper_2604_27158_gb300.train import fno_train_query
    kw = dict(c_in=4, c_out=1, width=width, layers=layers, modes=modes, dec_layers=1, dec_size=width)
    s, g = synth.FnoShape(**kw), FnoShape(**kw)
    p = torch.from_numpy(synth.fno_flatten_params(s, synth.fno_random_params(s, seed=5)).astype(np.float32)).cuda()
    x, dout = torch.randn((B, 4, H, W), device="cuda"), torch.randn((B, 1, H, W), device="cuda")
    out, dp = torch.empty_like(dout), torch.empty_like(p)
    sz, cfg = fno_train_query(g, B, H, W), g.c()
    saved = torch.empty(sz.saved_bytes // 4, device="cuda")
    ws = torch.empty(sz.ws_bytes + 256, dtype=torch.uint8, device="cuda")
    wp = ws.data_ptr() + (-ws.data_ptr()) % 256

    def once():
        call("fno_train_forward", ctypes.byref(cfg), p.data_ptr(), x.data_ptr(), out.data_ptr(), B, H, W,
             saved.data_ptr(), wp, _stream_ptr(None))
        call("fno_train_backward", ctypes.byref(cfg), p.data_ptr(), dout.data_ptr(), saved.data_ptr(), dp.data_ptr(),
             None, B, H, W, wp, _stream_ptr(None))

    once()
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        for _ in range(4):
            once()
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = float("inf")
    for _ in range(10):
        e[0].record()
        graph.replay()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) / 4)
    return best
