"""The adjoint step, the adjoint of the moments, moments and vorticity, each alone, against 64-bit
autograd (oracle/grad_oracle.py): random solids, every boundary kind, rows shorter than a lane's
chunk up to several row segments.  Batches that fill the chip with rows of whole 16-byte units take
the four-cells-a-lane kernels, the others the one-cell kernels; both are compared, and the two with
each other.  Bar: 2e-5 of the largest value (some hundred FP32 operations a cell, 6e-8 each)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import grad_oracle as go

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.lbm import GridSpec, Lattice  # noqa: E402

ALIGNED = [(4, 3), (8, 2), (28, 5), (32, 9), (124, 6), (128, 24), (132, 7), (256, 5), (260, 9), (512, 11)]
RAGGED = [(2, 2), (3, 4), (33, 7), (37, 6), (127, 5), (130, 6), (301, 8)]
FILLING = (640, 256)  # 163,840 cells: more than 1024 a multiprocessor
BAR = 2e-5


def _spec(nx, ny, kind, rng):
    solid = rng.random((ny, nx)) < 0.15
    if kind in ("pressure", "velocity"):
        solid[:, 0] = solid[:, -1] = False
        west = P.BC_PRESSURE if kind == "pressure" else P.BC_VELOCITY
        east = P.BC_PRESSURE if kind == "velocity" else P.BC_VELOCITY
        return GridSpec(nx, ny, 0.7, bc_west=west, bc_east=east, west_value=1.002 if kind == "pressure" else 0.03,
                        east_value=1.0 if kind == "velocity" else 0.02), solid
    return GridSpec(nx, ny, 0.8, **(dict(fx=1e-3, fy=-4e-4) if kind == "forced" else {})), solid


def _reference(grid, solid, state, mu, fields):
    """(adjoint step of mu, adjoint of the moments of `fields`, moments) at the shifted state, 64 bits."""
    tl = go.TorchLattice(oracle.Grid(nx=grid.nx, ny=grid.ny, tau=grid.tau, fx=grid.fx, fy=grid.fy,
                                     bc_west=grid.bc_west, bc_east=grid.bc_east, west_value=grid.west_value,
                                     east_value=grid.east_value), solid)
    gather = lambda f: torch.cat([f.reshape(-1), f.new_zeros(1)])[tl.pull_idx].reshape(9, grid.ny, grid.nx)
    g = gather(torch.from_numpy(state).double() + tl.w).requires_grad_(True)
    full = tl.boundary(g)
    step = torch.autograd.grad((gather(tl.collide(full)) * torch.from_numpy(mu)).sum(), g, retain_graph=True)[0]
    rho, ux, uy = tl.macro(full)
    seed = torch.autograd.grad(sum((a * torch.from_numpy(b)).sum() for a, b in zip((rho, ux, uy), fields)), g)[0]
    return step.numpy(), seed.numpy(), [v.detach().numpy() for v in (rho, ux, uy)]


def _off(t):
    """The same values at an address that is no multiple of 16 bytes."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    buf[1:] = t
    return buf[1:]


def _near(a, b, what):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    assert np.abs(a - b).max() <= BAR * max(np.abs(b).max(), 1e-3), what


@pytest.mark.parametrize("batch", ["small", "ragged", "filling", "filling_ragged"])
@pytest.mark.parametrize("kind", ["periodic", "forced", "pressure", "velocity"])
def test_adjoint_kernels_and_moments_match_fp64(kind, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(3)
    sizes = {"small": ALIGNED, "ragged": RAGGED, "filling": ALIGNED + [FILLING],
             "filling_ragged": RAGGED + ALIGNED + [FILLING]}[batch]
    specs = [_spec(nx, ny, kind, rng) for nx, ny in sizes]
    lat = Lattice([s[0] for s in specs], [s[1] for s in specs], u_max=0.9)
    n = lat.cells
    cells = torch.cat([torch.from_numpy(s[1].reshape(-1)) for s in specs]).cuda()
    solid9 = torch.cat([torch.from_numpy(np.broadcast_to(s[1], (9,) + s[1].shape).reshape(-1).copy())
                        for s in specs]).cuda()
    gen = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda m, sc: sc * torch.randn(m, generator=gen, device="cuda")
    state, mu = rnd(9 * n, 1e-2), rnd(9 * n, 1.0)
    state[solid9], mu[solid9] = 0.0, 0.0
    fields = [rnd(n, 1.0) for _ in range(3)]
    lat.set_state(state)
    step, seed, macro = lat.adjoint_step(state, mu), lat.adjoint_macro(state, *fields), lat.macro()
    # buffers at odd addresses take the one-cell kernel of the seed
    other = lat.adjoint_macro(_off(state), *fields)
    assert float((seed - other).abs().max()) <= BAR * float(other.abs().max())
    parts = [lat.split(t, 9) for t in (state, mu, step, seed)]
    fparts = [lat.split(t) for t in fields]
    mparts = [lat.split(t) for t in macro]
    for k, (grid, solid) in enumerate(specs):
        if (grid.nx, grid.ny) == FILLING:
            continue
        s, m, got_step, got_seed = [p[k].cpu().numpy() for p in parts]
        fs = [np.where(solid, 0.0, p[k].cpu().numpy().astype(np.float64)) for p in fparts]
        want_step, want_seed, want_macro = _reference(grid, solid, s, m.astype(np.float64), fs)
        _near(got_step, want_step, ("step", grid.nx, grid.ny))
        _near(got_seed, want_seed, ("seed", grid.nx, grid.ny))
        for a, b in zip(mparts, want_macro):
            _near(a[k].cpu().numpy(), b, ("moments", grid.nx, grid.ny))
    lat.close()


@pytest.mark.parametrize("kind", ["periodic", "pressure", "velocity"])
def test_vorticity_of_filling_batches(kind):
    """A chunk a lane (whole 16-byte rows) against the one-cell kernel at odd addresses, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(4)
    specs = [_spec(nx, ny, kind, rng) for nx, ny in ALIGNED + [FILLING]]
    lat = Lattice([s[0] for s in specs], [s[1] for s in specs], u_max=0.9)
    gen = torch.Generator(device="cuda").manual_seed(6)
    u = [0.02 * torch.randn(lat.cells, generator=gen, device="cuda") for _ in range(2)]
    assert torch.equal(lat.vorticity(*u), lat.vorticity(_off(u[0]), u[1]))
    lat.close()
