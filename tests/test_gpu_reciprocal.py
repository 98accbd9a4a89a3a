"""The reciprocal of the two-step passes: correctly rounded, so that their states are bitwise those of
single steps whatever the density."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2604_27158_gb300")
from paper_2604_27158_gb300._abi import call  # noqa: E402
from paper_2604_27158_gb300.lbm import GridSpec, Lattice, _stream_ptr  # noqa: E402


def _check(x):
    d = torch.from_numpy(x).cuda()
    y = torch.empty_like(d)
    call("lbm_reciprocal_eval", d.data_ptr(), y.data_ptr(), d.numel(), _stream_ptr(None))
    got = y.cpu().numpy()
    with np.errstate(all="ignore"):
        want = np.float32(1) / x
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.int32), want[~nan].view(np.int32))


def test_every_float_from_a_half_to_two():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _check((np.arange(1 << 24, dtype=np.uint32) + np.uint32(0x3F000000)).view(np.float32))


def test_floats_outside_the_range_alone_and_beside_others():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1)
    _check(rng.integers(0, 1 << 32, 1 << 20, dtype=np.uint64).astype(np.uint32).view(np.float32))
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, -1e-39, 1.1754944e-38, 3.4028235e38, -2e38, 0.49999997,
                     2.0, 2.0000002, -1.0, 0.25, 8.5e37], np.float32)
    x = rng.uniform(0.5, 2.0, (4 * edge.size, 4)).astype(np.float32)  # one outside value in each place of a lane
    for k in range(4):
        x[np.arange(edge.size) * 4 + k, k] = edge
    _check(x.ravel())
    _check(edge[:7].copy())  # a last thread with missing values


@pytest.mark.parametrize("kind", ["periodic", "forced", "open"])
def test_passes_equal_single_steps_for_densities_out_of_the_range(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(bc_west=P.BC_PRESSURE, bc_east=P.BC_PRESSURE, west_value=1.002) if kind == "open" else {}
    grid = GridSpec(132, 40, 0.8, fx=1e-5 if kind == "forced" else 0.0, **kw)
    solid = np.random.default_rng(2).random((40, 132)) < 0.1
    solid[:, 0] = solid[:, -1] = False
    gen = torch.Generator(device="cuda").manual_seed(5)
    state = torch.randn(9 * 132 * 40, generator=gen, device="cuda")
    for scale in (0.1, 0.4, 30.0):  # densities about 1 + 3 scale times a normal value
        out = []
        for passes in (True, False):
            lat = Lattice([grid], [solid], u_max=0.9)
            lat.set_passes(passes)
            lat.set_state(scale * state)
            rho = lat.macro()[0]
            assert float(rho.min()) < 0.5 and (scale < 0.3 or float(rho.max()) > 2)
            lat.step(4)
            out.append(lat.get_state())
            lat.close()
        a, b = out
        assert bool(((a == b) | (a.isnan() & b.isnan())).all()), scale
