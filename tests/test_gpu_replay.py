"""A captured lbm_step(n) with an even n can be replayed: the state must end in the buffer it
started from, whichever kernels take the steps.  Three replays, with other calls in between,
against the same steps outside a graph, bit for bit."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.fno import Fno, FnoShape, Hybrid, HybridConfig  # noqa: E402
from paper_2604_27158_gb300.lbm import GridSpec, Lattice  # noqa: E402

# batches that take two steps a pass, and one that steps singly (narrow rows that wrap in a chunk)
BATCHES = {"passes": [(128, 64)] * 3, "wide": [(512, 40)], "single": [(33, 30)] * 2}


def _lattice(sizes):
    rng = np.random.default_rng(4)
    solid = [rng.random((ny, nx)) < 0.1 for nx, ny in sizes]
    lat = Lattice([GridSpec(nx, ny, 0.8, fx=1e-6) for nx, ny in sizes], solid, u_max=0.9)
    parts = [synth.smooth_macro_fields(nx, ny, seed=k, drho=1e-3, umax=0.02) for k, (nx, ny) in enumerate(sizes)]
    lat.reinit(*[torch.from_numpy(np.concatenate([np.asarray(p[c], np.float32).ravel() for p in parts])).cuda()
                 for c in range(3)])
    return lat


def _capture(fn):
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        fn()
    return graph


@pytest.mark.parametrize("kind", list(BATCHES))
@pytest.mark.parametrize("n", [2, 4, 6, 50, 100])
def test_replayed_steps(kind, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, b = _lattice(BATCHES[kind]), _lattice(BATCHES[kind])
    graph = _capture(lambda: a.step(n))
    for between in (0, 6, 10):
        graph.replay()
        a.step(between)
        for _ in range(n + between):
            b.step(1)
        assert torch.equal(a.get_state(), b.get_state()), between
    a.close()
    b.close()


@pytest.mark.parametrize("k", [2, 6, 8])
def test_replayed_steps_between_hybrid_calls(k):
    """... also when unsteady cycles of k steps and steady solves run between the replays."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(c_in=4, c_out=3, width=16, layers=1, modes=4, dec_layers=1, dec_size=32)
    s = synth.FnoShape(**kw)
    net = Fno(FnoShape(**kw), synth.fno_flatten_params(s, synth.fno_random_params(s, seed=2)))
    states = []
    for replay in (True, False):
        lat = _lattice([(64, 32)] * 2)
        cycle = Hybrid(lat, net, HybridConfig(mode=1, k_lbm=k, m_fno=1, neq_mode=1))
        steady = Hybrid(lat, net, HybridConfig(mode=0, use_fno=0, check_every=5, tol=1e-12, max_steps=10 + k))
        graph = _capture(lambda: lat.step(4)) if replay else None
        for between in (lambda: cycle.advance(cycles=1), lambda: steady.advance(), lambda: cycle.advance(cycles=2)):
            graph.replay() if replay else lat.step(4)
            between()
        graph.replay() if replay else lat.step(4)
        states.append(lat.get_state())
        cycle.close()
        steady.close()
        lat.close()
    assert torch.equal(*states)
