"""The non-parallel arm of the paper's ablation (Sec. 4.2: every row in its own sensitivity order, against its own copy
of the inverse Hessian) through the C-ABI against the CPU oracle, on identical inputs; and its cost beside the
row-parallel method on the same layer."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_05576_b200 import ptq
from paper_2509_05576_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _run(W, H, Hinv, sc, zp, bits, mode):
    rows, cols = W.shape
    codes = torch.empty((rows, cols), dtype=torch.uint8, device="cuda")
    What = torch.empty((rows, cols), dtype=torch.float32, device="cuda")
    perm_rows = torch.full((rows, cols), -1, dtype=torch.int32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    st, ws = ptq.new_status(), ptq.Workspace()
    ptq.quantize_layer_per_row(_cuda(W), _cuda(Hinv), _cuda(sc), _cuda(zp), bits, mode, codes, What, perm_rows, _cuda(H),
                               loss, ws, st)
    torch.cuda.synchronize()
    ptq.check_status(st, "quantize_layer_per_row")
    return codes.cpu().numpy(), What.cpu().numpy(), perm_rows.cpu().numpy(), float(loss.item())


@pytest.mark.parametrize("rows,cols,n,bits", [(40, 128, 256, 4), (64, 64, 200, 3), (7, 33, 64, 8), (255, 128, 300, 4),
                                              (3, 1, 8, 4), (16, 108, 150, 4)])
@pytest.mark.parametrize("mode", [ptq.SCORE_QERR, ptq.SCORE_W | ptq.SCORE_ASCENDING])
def test_per_row_arm_matches_oracle(rows, cols, n, bits, mode):
    W, X = wl.make_layer(wl.LayerSpec("pr", rows, cols, n, bits, "kaiming", "halfnormal", 1400 + rows + cols))
    H = oracle.hessian_accumulate(X)
    Hinv, diag, _ = oracle.prepare_hinv(H)
    sc, zp = oracle.minmax_grid(W, bits)
    ref = oracle.quantize_layer_per_row(W, Hinv, diag, sc, zp, bits, mode, H_undamped=H)
    codes, What, perm_rows, loss = _run(W, H, Hinv, sc, zp, bits, mode)
    assert np.array_equal(perm_rows, ref["perm_rows"]), "a row's order differs"
    assert np.array_equal(codes, ref["codes"])
    assert np.array_equal(What, ref["What"])
    assert abs(loss - ref["loss"]) <= 1e-9 * ref["loss"]
    if rows > 1 and cols > 8:
        assert any(not np.array_equal(perm_rows[r], perm_rows[0]) for r in range(1, rows))   # the rows do differ


@pytest.mark.parametrize("rows,cols,bits", [(5, 8, 4), (3, 9, 3), (2, 7, 8), (2, 121, 4), (449, 127, 4)])
def test_per_row_arm_at_the_edges_of_its_tiles(rows, cols, bits):
    """Widths on and around the 8 x 8 tiles of the factorisation, and more rows than CTAs fit on the GPU at once."""
    W, X = wl.make_layer(wl.LayerSpec("pr", rows, cols, 2 * cols, bits, "kaiming", "normal", 1500 + rows + cols))
    H = oracle.hessian_accumulate(X)
    Hinv, diag, _ = oracle.prepare_hinv(H)
    sc, zp = oracle.minmax_grid(W, bits)
    ref = oracle.quantize_layer_per_row(W, Hinv, diag, sc, zp, bits, ptq.SCORE_QERR, H_undamped=H)
    codes, What, perm_rows, loss = _run(W, H, Hinv, sc, zp, bits, ptq.SCORE_QERR)
    assert np.array_equal(perm_rows, ref["perm_rows"])
    assert np.array_equal(codes, ref["codes"])
    assert np.array_equal(What, ref["What"])
    assert abs(loss - ref["loss"]) <= 1e-9 * ref["loss"]


def test_a_pivot_that_is_not_positive_is_reported():
    n = 20
    Hinv = np.eye(n)
    Hinv[11, 11] = -1.0
    W = np.full((1, n), 0.5, np.float32)
    with pytest.raises(ptq.PtqError) as ei:
        _run(W, np.eye(n), Hinv, np.ones(1, np.float32), np.zeros(1, np.float32), 4, ptq.SCORE_NONE)
    assert ei.value.code == ptq.ERR_NOT_SPD and "index 11" in str(ei.value)


@pytest.mark.parametrize("zero", [7.3, -0.5, 3.0e9, 1.0e17, -1.0e17])
def test_per_row_codes_follow_the_definition_for_any_zero_point(zero):
    """code = clamp(rint(w / s) + z, 0, maxq), q = s (code - z) in float64, also where z is no integer of ordinary size
    (identity: no compensation, so every weight is quantized as it stands)."""
    rng = np.random.Generator(np.random.PCG64(91))
    W = (rng.standard_normal((5, 20)) * 3.0).astype(np.float32)
    sc, zp = np.full(5, 0.25, np.float32), np.full(5, zero, np.float32)
    codes, What, _, _ = _run(W, np.eye(20), np.eye(20), sc, zp, 4, ptq.SCORE_NONE)
    z = zp[:, None].astype(np.float64)
    c = np.clip(np.rint(W.astype(np.float64) / 0.25) + z, 0.0, 15.0)
    assert np.array_equal(codes, c.astype(np.uint8))
    assert np.array_equal(What, (0.25 * (c - z)).astype(np.float32))


@pytest.mark.parametrize("pivot", [2.0e-308, 2.3e-308])
def test_pivots_on_either_side_of_the_normal_range(pivot):
    """1 / pivot is finite for both; nothing couples the columns, so every weight is rounded as it stands."""
    n = 11
    Hinv = np.eye(n)
    Hinv[4, 4] = pivot
    W = np.linspace(-1.0, 1.0, n, dtype=np.float32)[None, :].copy()
    codes, What, _, loss = _run(W, np.eye(n), Hinv, np.full(1, 0.125, np.float32), np.full(1, 8.0, np.float32), 4,
                                ptq.SCORE_NONE)
    c = np.clip(np.rint(W / 0.125) + 8.0, 0.0, 15.0)
    assert np.array_equal(codes, c.astype(np.uint8))
    assert np.isfinite(loss) and np.array_equal(What, (0.125 * (c - 8.0)).astype(np.float32))


def test_a_pivot_without_a_reciprocal_is_reported():
    n = 11
    Hinv = np.eye(n)
    Hinv[4, 4] = 1.0e-310
    with pytest.raises(ptq.PtqError) as ei:
        _run(np.full((1, n), 0.5, np.float32), np.eye(n), Hinv, np.ones(1, np.float32), np.zeros(1, np.float32), 4,
             ptq.SCORE_NONE)
    assert ei.value.code == ptq.ERR_NOT_SPD and "index 4" in str(ei.value)


def test_wider_layers_are_refused():
    fake = torch.zeros(16, dtype=torch.float32, device="cuda")
    st, ws = ptq.new_status(), ptq.Workspace()
    W = torch.zeros((4, 129), dtype=torch.float32, device="cuda")
    Hinv = torch.eye(129, dtype=torch.float64, device="cuda")
    codes = torch.empty((4, 129), dtype=torch.uint8, device="cuda")
    pr = torch.empty((4, 129), dtype=torch.int32, device="cuda")
    with pytest.raises(ptq.PtqError) as ei:
        ptq.quantize_layer_per_row(W, Hinv, fake, fake, 4, 0, codes, None, pr, None, None, ws, st)
    assert ei.value.code == ptq.ERR_UNSUPPORTED
