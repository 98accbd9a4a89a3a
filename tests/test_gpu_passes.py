"""Passes over two steps against single steps, with the choice set by hand: every row kind takes
both, also those that the estimate sends back to single steps.  Bitwise equal states."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300.lbm import GridSpec, Lattice, query_passes  # noqa: E402


def _spec(nx, ny, kind, seed):
    solid = np.random.default_rng(seed).random((ny, nx)) < 0.12
    if kind in ("open", "inlet"):
        solid[:, 0] = solid[:, -1] = False
        west = P.BC_PRESSURE if kind == "open" else P.BC_VELOCITY
        return GridSpec(nx, ny, 0.7, bc_west=west, bc_east=P.BC_PRESSURE, west_value=1.002 if kind == "open" else 0.03,
                        east_value=1.0), solid
    return GridSpec(nx, ny, 0.8, fx=1e-5 if kind == "forced" else 0.0), solid


def _lattice(specs, fields):
    lat = Lattice([s[0] for s in specs], [s[1] for s in specs], u_max=0.9)
    lat.reinit(*fields)
    return lat


def _fields(specs, seed, drho=1e-3):
    parts = [synth.smooth_macro_fields(g.nx, g.ny, seed=seed + k, drho=drho, umax=0.02) for k, (g, _) in enumerate(specs)]
    return [torch.from_numpy(np.concatenate([np.asarray(p[c], np.float32).ravel() for p in parts])).cuda()
            for c in range(3)]


# rows that wrap in a chunk, one to three chunks, strips of one, two and four warps with and without
# halo columns (484 and 490: two-warp strips of periodic rows)
SIZES = [(2, 2), (3, 5), (5, 7), (6, 3), (9, 2), (33, 12), (37, 21), (125, 6), (127, 6), (129, 4), (131, 9), (250, 5),
         (253, 7), (484, 6), (490, 11), (996, 3), (1021, 5), (1030, 4)]


@pytest.mark.parametrize("kind", ["periodic", "forced", "open", "inlet"])
def test_passes_equal_single_steps_on_rows_that_step_singly(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for sizes in [[s] for s in SIZES] + [SIZES, SIZES[::4] * 40, [(41, 60)] * 30]:
        specs = [_spec(nx, ny, kind, 3 * nx + ny + k) for k, (nx, ny) in enumerate(sizes)]
        fields = _fields(specs, 11)
        a, b = _lattice(specs, fields), _lattice(specs, fields)
        a.set_passes(True)
        b.set_passes(False)
        assert a.passes() and not b.passes()
        for n in (4, 9, 14):
            a.step(n)
            b.step(n)
            assert torch.equal(a.get_state(), b.get_state()), (kind, sizes[:3], n)
        assert a.steps_done() == b.steps_done() == 27
        a.close()
        b.close()


@pytest.mark.parametrize("kind", ["periodic", "forced", "open"])
def test_every_tile_shape_steps_singly(kind):
    """The single-step kernel of every tile shape, which passes would stand in for, against passes."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    specs = [_spec(nx, ny, kind, nx) for nx, ny in [(128, 33), (96, 64), (260, 11), (37, 25)]]
    fields = _fields(specs, 5)
    ref = _lattice(specs, fields)
    ref.set_passes(True)
    ref.step(13)
    for v in range(6):
        lat = _lattice(specs, fields)
        lat.set_passes(False)
        lat.set_step_variant(v)
        lat.step(13)
        assert torch.equal(lat.get_state(), ref.get_state()), v
        lat.close()
    ref.close()


@pytest.mark.parametrize("kind,nx,ny,n", [("forced", 90, 60, 31), ("periodic", 122, 120, 20), ("open", 32, 128, 19),
                                          ("periodic", 128, 128, 100), ("open", 512, 256, 20), ("forced", 128, 64, 1)])
def test_autotune_keeps_the_faster_of_passes_and_single_steps(kind, nx, ny, n):
    """... at batches where one takes at least 1.25 times as long as the other, which the estimate
    gets right as well; the state is unchanged."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    specs = [_spec(nx, ny, kind, 7)] * n
    lat = _lattice(specs, _fields(specs, 2))
    want = (nx, ny) in ((128, 128), (512, 256), (128, 64))
    assert lat.passes() == query_passes(lat.grids) == want
    before = lat.get_state()
    lat.set_passes(not want)
    lat.autotune(reps=3)
    assert lat.passes() == want and torch.equal(before, lat.get_state())
    lat.close()
