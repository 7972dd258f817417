"""The float64 product on the int8 tensor path (C += alpha A B^T from error-free slices; the product behind the deferred
part of Eq. 11) against a float64 library matmul, entry by entry, with the error bound of a float64 dot product."""
import numpy as np
import pytest
import torch

from paper_2509_05576_b200 import ptq

pytestmark = pytest.mark.gpu


def _run(m, n, k, b_is_kn, alpha, seed, scale_rows=False, ld_pad=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn((m, k + ld_pad), dtype=torch.float64, device="cuda", generator=g)[:, :k]
    Bs = (k, n + ld_pad) if b_is_kn else (n, k + ld_pad)
    Bf = torch.randn(Bs, dtype=torch.float64, device="cuda", generator=g)
    B = Bf[:, :n] if b_is_kn else Bf[:, :k]
    if scale_rows:
        A = A * torch.logspace(-6, 5, m, dtype=torch.float64, device="cuda")[:, None]
        A[min(3, m - 1)] = 0.0                                        # a dead row
        if not b_is_kn:
            B = B * torch.logspace(3, -4, n, dtype=torch.float64, device="cuda")[:, None]
        A = A.clone() if ld_pad == 0 else A
    C0 = torch.randn((m, n), dtype=torch.float64, device="cuda", generator=g)
    C = C0.clone()
    st, ws = ptq.new_status(), ptq.Workspace()
    ptq.gemm_nt_sliced(C, A, B, alpha, ws, st, b_is_kn=b_is_kn)
    torch.cuda.synchronize()
    ptq.check_status(st, "gemm_nt_sliced")
    Bt = B if b_is_kn else B.T
    ref = C0 + alpha * (A @ Bt)
    bound = 8e-16 * (A.abs() @ Bt.abs()) * abs(alpha) + 4e-16 * ref.abs() + 1e-300
    # entries far below a row's largest magnitude are rounded at 2^-55 of that magnitude: add that term
    bound = bound + abs(alpha) * k * 2.0 ** -54 * (A.abs().amax(dim=1)[:, None] * Bt.abs().amax(dim=0)[None, :])
    err = (C - ref).abs()
    assert bool((err <= bound).all()), float((err / bound).max())
    return float((err / (A.abs() @ Bt.abs() + 1e-300)).max())


@pytest.mark.parametrize("m,n,k", [(128, 64, 64), (300, 200, 500), (1, 1, 1), (257, 129, 1000), (70, 333, 96)])
@pytest.mark.parametrize("b_is_kn", [False, True])
def test_sliced_product_matches_float64_matmul(m, n, k, b_is_kn):
    rel = _run(m, n, k, b_is_kn, -1.0, 100 + m + n + k)
    assert rel < 1e-15          # relative to sum |a||b|: a float64 dot product's accuracy


def test_rows_of_very_different_magnitude_and_strided_operands():
    _run(200, 150, 320, False, 0.5, 7, scale_rows=True, ld_pad=8)
    _run(200, 150, 320, True, -2.0, 8, scale_rows=True, ld_pad=6)


def test_the_shape_of_a_deferred_update_of_a_tall_wide_layer():
    # rows x later-columns x super-block: several waves of tiles, many K blocks
    rel = _run(2048, 3000, 1024, True, -1.0, 9)
    assert rel < 1e-15


def _loss_launches():
    """Launches so far of the sliced int8 products and of the float64 product of the loss."""
    names = [ptq.lib().ptq_kernel_name(k).decode() for k in range(ptq.lib().ptq_kernel_count())]
    return np.array([ptq.launch_count(names.index(k)) for k in ("i8gemm_tcgen05", "dgemm_loss")])


def _loss_bound(D, H, loss):
    """Of a float64 product: independent rounding errors of up to u times a partial sum, sqrt(cols) of them per entry of
    dW H, three standard deviations of their weighted sum, and a few u for the last sums."""
    u = 2.0 ** -53
    return 3.0 * u * D.shape[1] ** 0.5 * torch.linalg.norm(D * (D.abs() @ H.abs())).item() + 4.0 * u * abs(float(loss))


@pytest.mark.parametrize("n,k", [(8, 1024), (65, 1024), (333, 1000), (40, 7)])
def test_columns_are_sliced_alike_in_one_pass_and_in_two(n, k):
    """Columns of up to 1024 values are cut into digits in one pass, longer ones in two.  With zeros below, the same columns
    go the other way: the product is the same bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(n + k)
    A = torch.randn((70, k), dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn((k, n + 3), dtype=torch.float64, device="cuda", generator=g)[:, :n]
    B *= torch.exp(3.0 * torch.randn(n, dtype=torch.float64, device="cuda", generator=g))
    out = []
    for rows in (k, 1025 + k):
        a, b = torch.zeros((70, rows), dtype=torch.float64, device="cuda"), torch.zeros((rows, n), dtype=torch.float64, device="cuda")
        a[:, :k], b[:k] = A, B
        C, st = torch.zeros((70, n), dtype=torch.float64, device="cuda"), ptq.new_status()
        ptq.gemm_nt_sliced(C, a, b, 1.0, ptq.Workspace(), st, b_is_kn=True)
        ptq.check_status(st)
        out.append(C)
    assert torch.equal(out[0], out[1])
    assert torch.allclose(out[0], A @ B, rtol=0.0, atol=1e-15 * float((A.abs() @ B.abs()).max()))


@pytest.mark.parametrize("rows,cols,sliced", [
    (512, 2304, True), (1000, 1791, True), (1400, 1400, True), (2600, 1024, True),     # above the line, the slices fit
    (560, 2304, False), (2561, 1025, False),                                           # above the line, they do not
    (505, 2304, False), (2430, 1050, False), (497, 2321, False)])                      # below the line
def test_loss_on_both_sides_of_the_line_between_its_products(rows, cols, sliced):
    """rows cols^2 just above and just below the line, odd widths among them, and sizes whose slices do not fit into what
    is free; both sums carry the rounding errors of a float64 product, hence twice the bound."""
    g = torch.Generator(device="cuda").manual_seed(rows)
    X = torch.randn((cols, cols + 64), device="cuda", generator=g).abs_()
    W = torch.randn((rows, cols), device="cuda", generator=g) * 0.03
    before = _loss_launches()
    b = ptq.quantize_layer_full(W, X, 4)
    torch.cuda.synchronize()
    ptq.check_status(b.status, "layer")
    assert ((_loss_launches() - before) > 0).tolist() == [sliced, not sliced]
    d = W.double() - b.What.double()
    want = 0.5 * float(((d @ b.H) * d).sum())
    assert abs(b.loss.item() - want) <= 2.0 * _loss_bound(d, b.H, want)


def _identity_layer(rows, cols, seed, hot):
    """W (float32) rounded as it stands (identity inverse Hessian) and a Hessian of normal activations; `hot` scales four
    input channels, whose weights are zero."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((cols, cols + cols // 2), dtype=torch.float64, device="cuda", generator=g)
    W = torch.randn((rows, cols), device="cuda", generator=g) * (2.0 / cols) ** 0.5
    if hot != 1.0:
        X[:4] *= hot
        W[:, :4] = 0.0
    H = 2.0 * (X @ X.T)
    return W, 0.5 * (H + H.T)


def _direct_loss(W, H):
    """The loss of ptq_quantize_layer, dW, the status word and how often the two products of the loss were launched."""
    rows, cols = W.shape
    st, ws = ptq.new_status(), ptq.Workspace()
    sc, zp = (torch.empty(rows, dtype=torch.float32, device="cuda") for _ in range(2))
    ptq.minmax_grid(W, 4, sc, zp, st)
    codes = torch.empty((rows, cols), dtype=torch.uint8, device="cuda")
    What = torch.empty((rows, cols), dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    before = _loss_launches()
    ptq.quantize_layer(W, torch.eye(cols, dtype=torch.float64, device="cuda"),
                       torch.arange(cols, dtype=torch.int32, device="cuda"), sc, zp, 4, codes, What, H, loss, ws, st)
    torch.cuda.synchronize()
    return loss.item(), W.double() - What.double(), st.tolist(), (_loss_launches() - before).tolist()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("rows,cols", [(512, 2304), (1000, 2048)])
def test_a_value_that_is_not_finite_in_the_hessian_shows_in_the_loss(rows, cols, value):
    W, H = _identity_layer(rows, cols, 5, 1.0)
    H[77, 1900] = H[1900, 77] = value
    loss, _, status, launches = _direct_loss(W, H)
    assert launches[0] > 0 and launches[1] == 0               # the sliced products
    assert not np.isfinite(loss)
    assert status[0] == ptq.ERR_NONFINITE


@pytest.mark.parametrize("value", [float("nan"), float("-inf")])
@pytest.mark.parametrize("b_is_kn", [False, True])
def test_a_value_that_is_not_finite_shows_in_its_row_or_column_of_the_product(b_is_kn, value):
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((130, 300), dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn((300, 70) if b_is_kn else (70, 300), dtype=torch.float64, device="cuda", generator=g)
    A[129, 299] = value
    B[(299, 65) if b_is_kn else (65, 299)] = value
    C = torch.zeros((130, 70), dtype=torch.float64, device="cuda")
    st, ws = ptq.new_status(), ptq.Workspace()
    ptq.gemm_nt_sliced(C, A, B, 1.0, ws, st, b_is_kn=b_is_kn)
    torch.cuda.synchronize()
    assert st.tolist()[0] == ptq.ERR_NONFINITE and st.tolist()[1] in (129, 65)
    bad = torch.zeros_like(C, dtype=torch.bool)
    bad[129], bad[:, 65] = True, True
    assert torch.equal(C.isnan(), bad) and bool(C[~bad].isfinite().all())


def _loss_in_two_doubles(D, H):
    """1/2 sum_ij D_ij (D H)_ij with every product and every sum carried as an unevaluated pair of doubles (Dekker's
    two-product, Knuth's two-sum): about 100 bits."""
    def split(x):
        t = x * 134217729.0
        hi = t - (t - x)
        return hi, x - hi
    Dh, Dl = split(D)
    Hh, Hl = split(H)
    s, c = torch.zeros_like(D), torch.zeros_like(D)
    for k in range(D.shape[1]):
        a, ah, al = D[:, k:k + 1], Dh[:, k:k + 1], Dl[:, k:k + 1]
        b, bh, bl = H[k:k + 1], Hh[k:k + 1], Hl[k:k + 1]
        p = a * b
        t = s + p
        z = t - s
        c += ((s - (t - z)) + (p - z)) + (((ah * bh - p) + ah * bl + al * bh) + al * bl)
        s = t
    s, c, D = (x.cpu().numpy().astype(np.longdouble) for x in (s, c, D))
    return 0.5 * np.sum((s + c) * D)


@pytest.mark.parametrize("rows,cols,hot", [(512, 2304, 1.0), (512, 2303, 1.0e5), (1000, 1791, 1.0e6)])
def test_loss_with_channels_of_very_different_scale(rows, cols, hot):
    W, H = _identity_layer(rows, cols, 6, hot)
    loss, D, status, launches = _direct_loss(W, H)
    assert status[0] == 0 and launches[0] > 0 and launches[1] == 0               # the sliced products
    want = _loss_in_two_doubles(D, H)
    bound = _loss_bound(D, H, want)
    assert abs(float(np.longdouble(loss) - want)) <= bound, (float((np.longdouble(loss) - want) / want), bound / float(want))


def _swept(rows, cols, channel_scale, damp, damp_mode, seed):
    """A layer whose input channels are scaled by `channel_scale`, through the sweep: its weights in the order of the sweep, and
    from the workspace, where they are the first arrays, the factor U, the weights as they were updated and the errors E."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((cols, cols + 512), device="cuda", generator=g) * channel_scale(cols, g)[:, None]
    W = torch.randn((rows, cols), device="cuda", generator=g) * (2.0 / cols) ** 0.5
    b, st, ws = ptq.LayerBuffers(rows, cols), ptq.new_status(), ptq.Workspace()
    ptq.hessian_accumulate(b.H.zero_(), X, ws, st)
    ptq.prepare_hinv(b.H, damp, damp_mode, b.Hinv, b.Hinv_diag, b.lam, ws, st)
    ptq.minmax_grid(W, 4, b.scale, b.zero, st)
    ptq.sensitivity_order(W, b.Hinv_diag, b.scale, b.zero, 4, ptq.SCORE_QERR, b.S, b.perm, ws, st)
    ws = ptq.Workspace()
    ptq.quantize_layer(W, b.Hinv, b.perm, b.scale, b.zero, 4, b.codes, b.What, None, None, ws, st)
    torch.cuda.synchronize()
    ptq.check_status(st)
    out, at = [], 0
    for m in (cols, rows, rows):
        out.append(ws.buf[at:at + 8 * m * cols].view(torch.float64).view(m, cols).cpu().numpy())
        at += (8 * m * cols + 255) // 256 * 256
    return W.double()[:, b.perm.long()].cpu().numpy(), *out


def _one_scale(cols, g):
    return torch.ones(cols, device="cuda")


def _log_normal(cols, g):
    return torch.exp(2.0 * torch.randn(cols, device="cuda", generator=g))


def _four_hot(cols, g):
    s = torch.ones(cols, device="cuda")
    s[torch.randperm(cols, device="cuda", generator=g)[:4]] = 1.0e4
    return s


@pytest.mark.parametrize("rows,cols", [(64, 3137), (33, 3200)])
@pytest.mark.parametrize("scale", [_one_scale, _log_normal, _four_hot])
@pytest.mark.parametrize("damp_mode,damp", [(ptq.DAMP_REL_MEAN_DIAG, 0.01), (ptq.DAMP_ABS, 0.01)])
def test_deferred_updates_are_as_exact_as_float64_steps(rows, cols, scale, damp_mode, damp):
    """W[:, later] -= E[:, panel] U[panel, later] of layers that are swept in panels of 1024 columns.  The first block of every
    later panel stays in memory as these products have left it: its error against extended precision, as root mean square of
    all and of each column, is no larger than that of float64 products of 64 columns each, subtracted one after the
    other (each rounds the weights once, and a panel's product once for all)."""
    W0, U, Wp, E = _swept(rows, cols, scale, damp, damp_mode, 40 + cols)
    for c0 in range(1024, cols, 1024):
        c1 = min(c0 + 64, cols)
        e, u = E[:, :c0], U[:c0, c0:c1]
        want = W0[:, c0:c1].astype(np.longdouble) - e.astype(np.longdouble) @ u.astype(np.longdouble)
        steps = W0[:, c0:c1].copy()
        for k in range(0, c0, 64):
            steps -= e[:, k:k + 64] @ u[k:k + 64]
        got, ref = ((a - want).astype(np.float64) ** 2 for a in (Wp[:, c0:c1], steps))
        assert got.mean() <= ref.mean(), (c0, (got.mean() / ref.mean()) ** 0.5)
        worst = (got.mean(axis=0) / ref.mean(axis=0)).max() ** 0.5
        assert worst <= 1.0, (c0, worst)
