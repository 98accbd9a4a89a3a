"""lbm_step's two-step passes against single steps: bitwise equal states for every kind of
row (one warp, groups of warps, strips with halo columns, wrapped and ragged ends), every
boundary kind, short task cuts and odd step counts."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.lbm import GridSpec, Lattice  # noqa: E402


def _spec(nx, ny, kind, seed):
    rng = np.random.default_rng(seed)
    solid = rng.random((ny, nx)) < 0.12
    if kind == "open":
        solid[:, 0] = solid[:, -1] = False
        return GridSpec(nx, ny, 0.7, bc_west=P.BC_PRESSURE, bc_east=P.BC_PRESSURE, west_value=1.002,
                        east_value=1.0), solid
    if kind == "inlet":
        return GridSpec(nx, ny, 0.6, bc_west=P.BC_VELOCITY, bc_east=P.BC_PRESSURE, west_value=0.03,
                        east_value=1.0), np.zeros_like(solid)
    return GridSpec(nx, ny, 0.8, fx=1e-5 if kind == "forced" else 0.0), solid


def _fields(specs, seed):
    parts = [synth.smooth_macro_fields(g.nx, g.ny, seed=seed + k, drho=1e-3, umax=0.02)
             for k, (g, _) in enumerate(specs)]
    return [torch.from_numpy(np.concatenate([np.asarray(p[c], np.float32).ravel() for p in parts])).cuda()
            for c in range(3)]


SIZES = [(2, 2), (3, 5), (4, 3), (5, 7), (8, 2), (37, 21), (124, 9), (125, 6), (127, 6), (128, 64),
         (129, 4), (132, 5), (248, 11), (256, 40), (260, 3), (301, 23), (384, 7), (504, 5), (512, 70),
         (513, 9), (516, 8), (700, 6), (1021, 5), (1500, 9)]


@pytest.mark.parametrize("kind", ["periodic", "forced", "open", "inlet"])
def test_passes_equal_single_steps_for_every_row_length(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for group in ([s] for s in SIZES), [SIZES], [SIZES[::5] * 40]:
        for sizes in group:
            specs = [_spec(nx, ny, kind, 7 * nx + ny + k) for k, (nx, ny) in enumerate(sizes)]
            fields = _fields(specs, 11)
            a = Lattice([s[0] for s in specs], [s[1] for s in specs], u_max=0.9)
            b = Lattice([s[0] for s in specs], [s[1] for s in specs], u_max=0.9)
            a.reinit(*fields)
            b.reinit(*fields)
            for n in (2, 3, 8):
                a.step(n)
                for _ in range(n):
                    b.step(1)
                assert torch.equal(a.get_state(), b.get_state()), (kind, sizes[:3], n)
            assert a.steps_done() == b.steps_done() == 13
            a.close()
            b.close()
