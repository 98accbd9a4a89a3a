"""CPU-side checks of the C ABI: the library builds, loads, exports every declared
symbol, and validates arguments on the host (no GPU work is issued)."""
import ctypes

import numpy as np
import pytest

import paper_2604_27158_gb300 as P
from paper_2604_27158_gb300 import _abi
from paper_2604_27158_gb300.lbm import GridSpec, query_layout


def test_library_exports_every_declared_symbol():
    lib = P.lib()
    names = _abi.declared_symbols()
    assert len(names) >= 12
    for n in names:
        assert hasattr(lib, n), n


def test_query_layout_sizes():
    grids = [GridSpec(128, 64, 0.8), GridSpec(37, 20, 0.6, bc_west=P.BC_PRESSURE,
                                                bc_east=P.BC_PRESSURE, west_value=1.001)]
    lay = query_layout(grids)
    assert lay.cells == 128 * 64 + 37 * 20
    assert lay.f_elems == 9 * (64 * 128 + 20 * 64)       # pitch = nx rounded up to 32
    assert lay.mask_words == 64 * 4 + 20 * 2
    assert lay.ws_bytes > 0 and lay.ws_bytes % 256 == 0


@pytest.mark.parametrize("bad", [
    GridSpec(1, 8, 0.8),                                   # too small
    GridSpec(8, 8, 0.5),                                   # tau must exceed 1/2
    GridSpec(8, 8, 0.8, bc_west=P.BC_PRESSURE),            # periodic on one end only
    GridSpec(8, 8, 0.8, bc_west=P.BC_VELOCITY, bc_east=P.BC_PRESSURE, west_value=0.7),
    GridSpec(8, 8, 0.8, bc_west=7, bc_east=7),
])
def test_query_layout_rejects_invalid_grids(bad):
    with pytest.raises(P.LbmError) as e:
        query_layout([bad])
    assert e.value.code == _abi.LBM_ERR_INVALID_ARG
    assert "lbm" in str(e.value)


def test_null_arguments_rejected_without_gpu():
    lib = P.lib()
    assert lib.lbm_query_layout(None, 0, None) == _abi.LBM_ERR_INVALID_ARG
    h = ctypes.c_void_p()
    assert lib.lbm_init(None, 0, None, None, None, None, 0.2, None, ctypes.byref(h)) == _abi.LBM_ERR_INVALID_ARG
    assert lib.lbm_step(None, 1, None) == _abi.LBM_ERR_INVALID_ARG
    assert h.value is None


def test_mask_packing_layout():
    solid = np.zeros((3, 40), bool)
    solid[1, 33] = True
    solid[2, 0] = True
    w = P.pack_mask(solid)
    assert w.shape == (6,)
    assert w[1 * 2 + 1] == (1 << 1) and w[2 * 2] == 1 and w.sum() == 3


def test_fno_query_counts_the_papers_parameters():
    """The library's parameter layout (fno_query, host only) has exactly the totals the
    paper prints for its six model shapes."""
    import json
    import os
    from paper_2604_27158_gb300.fno import FnoShape, fno_query
    with open(os.path.join(os.path.dirname(__file__), "golden", "fno_param_counts.json")) as fh:
        models = json.load(fh)["models"]
    for mdl in models:
        shape = FnoShape(c_in=mdl["c_in"], c_out=mdl["c_out"], width=mdl["width"],
                         layers=mdl["layers"], modes=mdl["modes"], dec_layers=mdl["dec_layers"],
                         dec_size=mdl["dec_size"])
        sz = fno_query(shape, 1, 2 * mdl["modes"], 2 * mdl["modes"] + 1)
        assert sz.n_params == mdl["params"], mdl["name"]
        assert sz.packed_bytes % 256 == 0 and sz.ws_bytes > 0


@pytest.mark.parametrize("kw,B,H,W", [
    (dict(modes=8), 1, 15, 64),      # 2m > H
    (dict(modes=8), 1, 32, 16),      # m >= W / 2
    (dict(width=15), 1, 32, 32),     # odd width
    (dict(width=66), 1, 32, 32),     # width above 64
    (dict(activation=5), 1, 32, 32),
])
def test_fno_query_rejects_invalid_shapes(kw, B, H, W):
    from paper_2604_27158_gb300.fno import FnoShape, fno_query
    with pytest.raises(P.LbmError) as e:
        fno_query(FnoShape(**kw), B, H, W)
    assert e.value.code == _abi.LBM_ERR_INVALID_ARG


def test_hybrid_workspace_holds_every_group_and_network():
    """An FNO step runs its size groups, and the two networks of a group, as parallel
    branches, so no two of them may share FNO buffers: the hybrid workspace (a host-only
    query) grows by at least the FNO workspaces of both networks when a size group is
    added, and holds those of every (group, network) pair."""
    from paper_2604_27158_gb300._abi import call, lbm_grid
    from paper_2604_27158_gb300.fno import FnoShape, fno_query
    sr = FnoShape(c_in=1, c_out=1, width=16, layers=2, modes=4, dec_size=32)
    su = FnoShape(c_in=2, c_out=2, width=16, layers=2, modes=8, dec_size=32)

    def ws(grids):
        arr = (lbm_grid * len(grids))(*[g.c() for g in grids])
        n = ctypes.c_size_t()
        fc, fcu = sr.c(), su.c()
        call("hybrid_query_ws", arr, len(grids), ctypes.byref(fc), ctypes.byref(fcu),
             ctypes.byref(n))
        return n.value

    one = [GridSpec(128, 64, 0.8)] * 3
    two = one + [GridSpec(96, 48, 0.7)] * 2
    fno_ws = {(B, H, W): fno_query(sr, B, H, W).ws_bytes + fno_query(su, B, H, W).ws_bytes
              for B, H, W in ((3, 64, 128), (2, 48, 96))}
    assert ws(one) >= fno_ws[(3, 64, 128)]
    assert ws(two) - ws(one) >= fno_ws[(2, 48, 96)]
    assert ws(two) >= sum(fno_ws.values())


@pytest.mark.parametrize("act", [0, 1])
def test_training_refuses_misaligned_saved_activations(act):
    """saved_d holds complex pairs: a buffer that is not 8-byte aligned is refused on the host,
    by either call, before anything is launched (the pointers here are never read)."""
    from paper_2604_27158_gb300.fno import FnoShape
    cfg = FnoShape(width=8, layers=1, modes=2, dec_size=8, activation=act).c()
    lib, p = _abi.lib(), 4096
    for off in (1, 4, 12):
        assert lib.fno_train_forward(ctypes.byref(cfg), p, p, p, 1, 8, 8, p + off, p, None) == _abi.LBM_ERR_INVALID_ARG
        assert lib.fno_train_backward(ctypes.byref(cfg), p, p, p + off, p, None, 1, 8, 8, p,
                                      None) == _abi.LBM_ERR_INVALID_ARG


# (kind, nx, ny, grids) and the measured time of two single steps over that of one pass
MEASURED_PASSES = [
    ("forced", 90, 60, 31, 0.74), ("forced", 293, 219, 3, 0.77), ("forced", 55, 78, 27, 0.78),
    ("free", 122, 120, 20, 0.78), ("free", 65, 149, 14, 0.79), ("forced", 110, 152, 16, 0.77),
    ("free", 130, 60, 16, 0.83), ("free", 54, 67, 32, 0.83), ("forced", 130, 64, 10, 0.85),
    ("open", 32, 128, 19, 0.76), ("open", 36, 68, 30, 0.81), ("open", 33, 65, 34, 0.86),
    ("forced", 180, 119, 8, 0.89), ("forced", 255, 100, 22, 0.85), ("forced", 193, 156, 5, 0.88),
    ("forced", 128, 64, 1, 1.47), ("open", 512, 256, 64, 1.7), ("open", 4096, 4096, 1, 1.5),
    ("open", 512, 256, 20, 1.6), ("free", 128, 128, 100, 1.7), ("free", 64, 64, 1, 1.44),
    ("forced", 256, 128, 46, 1.56), ("free", 512, 100, 23, 1.46), ("forced", 621, 273, 12, 1.14),
    ("free", 139, 79, 87, 1.43), ("open", 262, 139, 18, 1.4), ("free", 48, 48, 1, 1.5)]


@pytest.mark.parametrize("kind,nx,ny,n,gain", MEASURED_PASSES)
def test_passes_are_estimated_to_pay_where_they_do(kind, nx, ny, n, gain):
    """lbm_step takes two steps a pass by an estimate that is a function of the batch alone; at
    batches with a clear outcome it agrees with the measurement."""
    from paper_2604_27158_gb300.lbm import query_passes
    kw = dict(bc_west=P.BC_PRESSURE, bc_east=P.BC_PRESSURE, west_value=1.001) if kind == "open" else {}
    grid = GridSpec(nx, ny, 0.7, fx=1e-6 if kind == "forced" else 0.0, **kw)
    assert query_passes([grid] * n) == (gain > 1)
