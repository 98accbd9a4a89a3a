"""The four-cells-a-lane kernels against the one-cell kernels they stand in for: the same call
with buffers that are not 16-byte aligned takes the general kernels.  Every boundary kind, rows
shorter than a warp, exactly one, and several segments, disks everywhere.  Copies and stencils
are equal; the adjoint kernels may contract other products (FP32 rounding: 2e-6 of the largest)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.lbm import GridSpec, Lattice  # noqa: E402

SIZES = [(4, 3), (8, 2), (28, 5), (32, 9), (124, 6), (128, 64), (132, 7), (256, 5), (260, 9), (512, 33)]


def _lattice(kind, sizes, seed):
    rng = np.random.default_rng(seed)
    grids, masks = [], []
    for nx, ny in sizes:
        solid = rng.random((ny, nx)) < 0.15
        if kind == "periodic":
            grids.append(GridSpec(nx, ny, 0.8, fx=1e-5))
        else:
            solid[:, 0] = solid[:, -1] = False
            west = P.BC_PRESSURE if kind == "pressure" else P.BC_VELOCITY
            grids.append(GridSpec(nx, ny, 0.7, bc_west=west, bc_east=P.BC_PRESSURE,
                                  west_value=1.002 if kind == "pressure" else 0.03, east_value=1.0))
        masks.append(solid)
    return Lattice(grids, masks, u_max=0.9)


def _off(t):
    """The same values at an address that is no multiple of 16 bytes."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    buf[1:] = t
    return buf[1:]


@pytest.mark.parametrize("kind", ["periodic", "pressure", "velocity"])
def test_chunk_kernels_equal_cell_kernels(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for sizes in [[s] for s in SIZES] + [SIZES]:
        lat = _lattice(kind, sizes, 3)
        gen = torch.Generator(device="cuda").manual_seed(5)
        rnd = lambda n, s: s * torch.randn(n, generator=gen, device="cuda")
        state, mu = rnd(9 * lat.cells, 1e-2), rnd(9 * lat.cells, 1.0)
        fields = [rnd(lat.cells, 0.02) for _ in range(3)]
        lat.set_state(state)
        a = lat.get_state()
        lat.set_state(_off(state))
        assert torch.equal(a, lat.get_state()) and torch.equal(a, state)
        assert torch.equal(lat.vorticity(*fields[:2]), lat.vorticity(_off(fields[0]), fields[1]))

        def near(x, y):
            return float((x - y).abs().max()) <= 2e-6 * float(y.abs().max())

        assert near(lat.adjoint_step(state, mu), lat.adjoint_step(_off(state), _off(mu), out=_off(mu)))
        assert near(lat.adjoint_macro(state, *fields), lat.adjoint_macro(_off(state), *fields))
        # moments of the pull against the exported populations (another kernel)
        rho, ux, _ = lat.macro()
        for k, (g, ex, r, u) in enumerate(zip(lat.grids, lat.split(lat.export_f(), 9), lat.split(rho), lat.split(ux))):
            solid = torch.from_numpy(lat.solid[k]).cuda()
            want = torch.where(solid, torch.ones_like(r), 1 + ex.double().sum(0).float())
            assert float((r - want).abs().max()) < 1e-6
            assert bool((u[solid] == 0).all())
        lat.close()


@pytest.mark.parametrize("kind", ["periodic", "pressure", "velocity"])
def test_small_and_large_batches_agree(kind):
    """Moments and their adjoint of small batches (a cell a thread) against the same grids beside
    one that fills the chip (a chunk a lane, SIZES + 163,840 cells); vorticity of single grids
    likewise.  FP32 rounding: 2e-6 of the largest."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sizes = SIZES + [(33, 7), (127, 5), (130, 6)] if kind != "pressure" else SIZES
    small, large = _lattice(kind, sizes, 3), _lattice(kind, sizes + [(640, 256)], 3)
    n = small.cells
    assert n < 100_000
    gen = torch.Generator(device="cuda").manual_seed(5)
    state = 1e-2 * torch.randn(9 * large.cells, generator=gen, device="cuda")
    fields = [0.02 * torch.randn(large.cells, generator=gen, device="cuda") for _ in range(3)]
    small.set_state(state[:9 * n])
    large.set_state(state)

    def near(x, y):
        return float((x - y).abs().max()) <= 2e-6 * float(y.abs().max())

    for a, b in zip(small.macro(), large.macro()):
        assert near(a, b[:n])
    a = small.adjoint_macro(state[:9 * n], *[f[:n] for f in fields])
    assert near(a, large.adjoint_macro(state, *fields)[:9 * n])
    omega = large.vorticity(*fields[:2])
    for k, w in enumerate(large.split(omega)[:len(sizes)]):
        one = Lattice([large.grids[k]], [large.solid[k]], u_max=0.9)
        u = [large.split(f)[k].reshape(-1).contiguous() for f in fields[:2]]
        assert torch.equal(one.vorticity(*u), w.reshape(-1))
        one.close()
    small.close()
    large.close()
