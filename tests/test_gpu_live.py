"""Dense plans on a scene grid skip the zero columns beyond the last library
radius: results against the oracle at the edges of the skipping (odd and tiny
grids, groups cut by rows, no live column at all), and a non-finite scene or
residual value at a skipped column still makes the result NaN."""
import numpy as np
import pytest
import torch

from oracle import psfsim_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GRIDS = [(1, 0.5, 3.0), (7, 1.0, 2.0), (31, 0.5, 3.0), (64, 0.5, 4.0), (65, 0.3, 4.0), (90, 0.25, 2.6), (96, 0.5, 1.0),
         (12, 1.0, 0.2)]  # N, S, last radius; the last has no pixel inside


def _plan(N, S, r_last, storage, n=20, n_r=5, seed=5):
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(seed)
    radii = np.linspace(0.0, r_last, n_r)
    lib = rng.uniform(0.0, 1.0, (n_r, n, n)).astype(np.float32)
    plan = Plan(torch.from_numpy(lib).to(DEV), radii, 0.25, N=N, S=S, storage=storage)
    return plan, O.build_A(lib.astype(np.float64), radii, N, S), rng


def _check_forward(plan, A, x, tol, **kw):
    y = plan.forward(torch.from_numpy(x).to(DEV), **kw).double().cpu().numpy()
    x64 = x.astype(np.float64)
    err = O.bound_relative_error(y, x64 @ A.T, x64 @ np.abs(A).T, floor=O.FLT_MIN).max()
    assert err <= tol and plan.sync_status() == 0, err


@pytest.mark.parametrize("storage,tol", [("split_bf16", 1e-5), ("bf16", 2.0 ** -8 + 2.5e-5), ("fp32", 1e-5)])
@pytest.mark.parametrize("N,S,r_last", GRIDS)
def test_forward_skips_only_zero_columns(N, S, r_last, storage, tol):
    plan, A, rng = _plan(N, S, r_last, storage)
    _check_forward(plan, A, rng.uniform(0.0, 1.0, (3, N * N)).astype(np.float32), tol)


@pytest.mark.parametrize("B", [1, 2, 4, 5, 8, 9, 12, 13, 16, 17, 33])
@pytest.mark.parametrize("storage", ["fp32", "fp32_sym"])
def test_fp32_forward_batches(B, storage):
    """Every group width of the batched product, its remainders, and the filter for zero pixels;
    an odd image (row quads cut at the end), more than one 256-column chunk per share."""
    plan, A, rng = _plan(64, 0.125, 4.0, storage, n=17)
    x = rng.uniform(0.0, 1.0, (B, 64 * 64)).astype(np.float32)
    x[:, rng.uniform(size=64 * 64) < 0.7] = 0.0
    _check_forward(plan, A, x, 1e-5)
    if storage == "fp32":
        _check_forward(plan, A, x, 1e-5, skip_zeros=True)


@pytest.mark.parametrize("storage,kw", [("split_bf16", {}), ("bf16", {}), ("fp32", {}), ("fp32", {"skip_zeros": True})])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_scene_value_at_a_skipped_column(storage, kw, value):
    plan, A, rng = _plan(64, 0.5, 4.0, storage)
    dead = np.nonzero(~A.any(axis=0))[0]
    for j in (dead[0], dead[len(dead) // 2], dead[-1]):
        x = rng.uniform(0.0, 1.0, (2, 64 * 64)).astype(np.float32)
        x[1, j] = value
        y = plan.forward(torch.from_numpy(x).to(DEV), **kw).cpu().numpy()
        assert np.isfinite(y[0]).all() and np.isnan(y[1]).all()
        y = plan.forward(torch.from_numpy(x[1]).to(DEV), **kw).cpu().numpy()
        assert np.isnan(y).all()


@pytest.mark.parametrize("storage", ["split_bf16", "bf16"])
@pytest.mark.parametrize("n,N,interp", [(17, 48, "linear"), (96, 64, "linear"), (41, 50, "nearest"), (33, 66, "linear"),
                                        (24, 320, "linear"), (20, 150, "linear")])
def test_pixelwise_build_equals_direct_build_bit_for_bit(n, N, interp, storage):
    """Dense split builds of an even grid (odd images, runs of 8 and ragged runs) against the
    same grid given as field points, which takes the direct build; padding is zero."""
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(n * N)
    radii, S = np.linspace(0.0, 5.0, 4), 8.0 / N
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (4, n, n)).astype(np.float32)).to(DEV)
    c = (np.arange(N) - 0.5 * (N - 1)) * S
    pts = np.stack([np.tile(c, N), np.repeat(c, N)], axis=1)
    grid = Plan(lib, radii, 0.25, N=N, S=S, storage=storage, interp=interp)
    direct = Plan(lib, radii, 0.25, points=pts, storage=storage, interp=interp)
    for a, b in zip(grid.A_split(), direct.A_split()):
        assert (a is None) == (b is None)
        if a is not None:
            assert torch.equal(a.view(torch.int16 if a.dtype == torch.bfloat16 else torch.int32),
                               b.view(torch.int16 if b.dtype == torch.bfloat16 else torch.int32))


def test_split_build_in_a_workspace_without_room_for_pair_entries():
    """A workspace of the layout's size alone is enough: the block-wise build, the same bits."""
    import ctypes
    from paper_2106_09122_gb300 import Plan
    from paper_2106_09122_gb300 import _binding as B
    n, N, n_r = 33, 66, 4
    rng = np.random.default_rng(3)
    radii, S = np.linspace(0.0, 5.0, n_r), 8.0 / N
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (n_r, n, n)).astype(np.float32)).to(DEV)
    plan = Plan(lib, radii, 0.25, N=N, S=S, storage="split_bf16")
    up = lambda v: (v + 255) // 256 * 256
    extra = up(((n_r - 1) * (n + 1) ** 2 + 1) * 32) + up(n * n * 4)
    ws = torch.zeros(plan.workspace.numel() - extra, dtype=torch.uint8, device=DEV)
    h, L = ctypes.c_void_p(), B.load()
    args = (ctypes.c_void_p(lib.data_ptr()), radii.ctypes.data_as(ctypes.c_void_p), n_r, n, 0.25, N, S,
            B.SPLIT_BF16, B.LINEAR, ctypes.c_void_p(ws.data_ptr()))
    assert L.psfsim_build(*args, ws.numel() - 256, None, ctypes.byref(h)) == B.ERR_WORKSPACE
    B.check(L.psfsim_build(*args, ws.numel(), None, ctypes.byref(h)), "psfsim_build")
    torch.cuda.synchronize()
    end = plan.info.scale_offset + 4 * plan.info.ld
    assert torch.equal(ws[:end], plan.workspace[:end])
    L.psfsim_free(h)


ADJOINT_TOL = {"fp32": 1e-5, "fp32_sym": 1e-5, "split_bf16": 1e-5, "split_bf16_sym": 1e-5, "bf16": 2.0 ** -8 + 1e-5}


@pytest.mark.parametrize("storage,B", [("fp32", b) for b in (1, 2, 4, 5, 8, 9, 16, 17)] + [("fp32_sym", 1), ("fp32_sym", 3)] +
                         [(s, b) for s in ("split_bf16", "bf16") for b in (1, 16, 17, 33, 80, 81)] +
                         [("split_bf16_sym", b) for b in (1, 5, 21)])
@pytest.mark.parametrize("n,N,S,r_last", [(20, 31, 0.5, 3.0), (17, 64, 0.5, 4.0), (33, 40, 0.25, 6.0), (20, 12, 1.0, 0.2)])
def test_adjoint_reads_only_live_columns(storage, B, n, N, S, r_last):
    """Odd images (row quads cut at the end), more than one 64-column range per CTA or fewer
    columns than CTAs, no live column at all; a column beyond the last radius is exactly zero."""
    if storage.endswith("_sym") and N % 2:
        pytest.skip("an even scene grid")
    plan, A, rng = _plan(N, S, r_last, storage, n=n)
    g = rng.standard_normal((B, n * n)).astype(np.float32)
    gx = plan.adjoint(torch.from_numpy(g).to(DEV)).double().cpu().numpy()
    g64 = g.astype(np.float64)
    err = O.bound_relative_error(gx, g64 @ A, np.abs(g64) @ np.abs(A), floor=O.FLT_MIN).max()
    assert err <= ADJOINT_TOL[storage] and plan.sync_status() == 0, err
    assert np.all(gx[:, ~A.any(axis=0)] == 0.0)


@pytest.mark.parametrize("storage", ["fp32", "split_bf16", "bf16"])
@pytest.mark.parametrize("B", [1, 3, 9])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_residual_comes_out_as_multiplied_out(storage, B, value):
    """An infinite residual value gives an infinity where its element of A is not zero, and NaN
    (0 x inf) where it is: also in the columns that are not read."""
    plan, A, rng = _plan(64, 0.5, 4.0, storage)
    for i in (0, 211, 399):
        g = rng.standard_normal((B, 400)).astype(np.float32)
        g[B - 1, i] = value
        gx = plan.adjoint(torch.from_numpy(g).to(DEV)).cpu().numpy()
        assert np.isfinite(gx[:B - 1]).all()
        with np.errstate(invalid="ignore"):
            want = np.where(A[i] == 0.0, np.nan, value * np.sign(A[i]))
        assert np.array_equal(gx[B - 1], want.astype(np.float32), equal_nan=True)


@pytest.mark.parametrize("n,N,S,r_last", [(20, 31, 0.5, 3.0), (17, 64, 0.5, 4.0), (32, 96, 0.5, 2.0), (21, 12, 1.0, 0.2)])
def test_ring_gradient_reads_only_live_columns(n, N, S, r_last):
    """The fused gradient against the separate operators: rings that reach beyond the last
    radius, few or no live columns, odd images; zero gradient at the columns not read."""
    from paper_2106_09122_gb300.fit import RingProblem
    plan, A, rng = _plan(N, S, r_last, "fp32", n=n)
    target = torch.from_numpy((rng.uniform(0.5, 1.5, n * n) * 1e-9).astype(np.float32)).to(DEV)
    P = RingProblem(plan, N, S, 1.5 * r_last, target, 1e-11)
    assert P.fused
    theta = np.array([1.1 * r_last, r_last / 2, np.deg2rad(40.0), 0.3, 1e-9])
    loss, grad = P.loss_and_grad(theta)
    y, gz, z = P.y.clone(), P.gz.clone(), P.z.clone()
    loss2, grad2 = P.loss_and_grad(theta)
    assert loss2 == loss and np.array_equal(grad2, grad)
    assert torch.all(gz[torch.from_numpy(~A.any(axis=0)).to(DEV)] == 0)
    P.fused = False
    loss_s, grad_s = P.loss_and_grad(theta)
    assert torch.equal(P.z, z)
    assert torch.allclose(P.y, y, rtol=1e-6, atol=0) and torch.allclose(P.gz, gz, rtol=1e-5, atol=1e-5 * float(gz.abs().max()))
    assert loss == pytest.approx(loss_s, rel=1e-6)
    np.testing.assert_allclose(grad, grad_s, rtol=1e-5, atol=1e-6 * np.abs(grad_s).max())


def test_ring_gradient_with_a_target_that_is_not_finite():
    from paper_2106_09122_gb300.fit import RingProblem
    plan, A, rng = _plan(64, 0.5, 4.0, "fp32")
    target = torch.full((400,), 1e-9, device=DEV)
    target[123] = float("nan")
    P = RingProblem(plan, 64, 0.5, 4.0, target, 1e-11)
    loss, grad = P.loss_and_grad(np.array([2.0, 1.0, 0.5, 0.3, 1e-9]))
    assert np.isnan(loss) and np.isnan(grad).all() and torch.isnan(P.gz).all() and torch.isfinite(P.y).all()


@pytest.mark.parametrize("storage,tol,B", [(s, t, b) for s, t in (("split_bf16", 1e-5), ("bf16", 2.0 ** -8 + 2.5e-5))
                                           for b in (81, 100, 128, 129, 200, 256)] +
                         [("split_bf16_sym", 1e-5, b) for b in (20, 21, 32, 33, 50, 64)])
@pytest.mark.parametrize("n", [17, 24])
def test_forward_of_many_scenes(storage, tol, B, n):
    """Around the batch where scenes become the product's rows: partial blocks of 128, images
    that end inside a tile of 256 pixels, skipped k-tiles."""
    plan, A, rng = _plan(64, 0.125, 3.0, storage, n=n)
    _check_forward(plan, A, rng.uniform(0.0, 1.0, (B, 64 * 64)).astype(np.float32), tol)


@pytest.mark.parametrize("storage,tol", [("split_bf16", 1e-5), ("bf16", 2.0 ** -8 + 2.5e-5)])
@pytest.mark.parametrize("units", [0, 1, 2, 40])
@pytest.mark.parametrize("n,shift", [(17, 0), (33, 0), (32, 0), (32, 1), (40, 2)])
def test_sum_over_splits(storage, tol, units, n, shift):
    """One job's k-splits from none to more than 8 (both forms of their sum), into images whose
    rows start at any 4-byte address, ending inside a thread's 4 rows and inside a CTA's 1024."""
    from paper_2106_09122_gb300.serve import MultiForward
    plan, A, rng = _plan(64, 0.125, 3.0, storage, n=n)
    x = rng.uniform(0.0, 1.0, (5, 64 * 64)).astype(np.float32)
    big = torch.full((5 * plan.M + 8,), float("nan"), device=DEV)
    y = big[shift:shift + 5 * plan.M].view(5, plan.M)
    mf = MultiForward([plan], [5], tuning=(0, units, 0) if units else None, y=[y])
    mf.x[0].copy_(torch.from_numpy(x))
    mf.count.fill_(4)
    mf.enqueue()
    x64 = x[:4].astype(np.float64)
    err = O.bound_relative_error(y[:4].double().cpu().numpy(), x64 @ A.T, x64 @ np.abs(A).T, floor=O.FLT_MIN).max()
    assert err <= tol and plan.sync_status() == 0, err
    assert torch.isnan(big[:shift]).all() and torch.isnan(big[shift + 4 * plan.M:]).all()


@pytest.mark.parametrize("n", [251, 252])
def test_sum_over_splits_of_many_rows(n):
    """More than four splits summed by one thread (many rows): against one and two splits, each
    within 1e-5 of sums of products that are not negative."""
    from paper_2106_09122_gb300 import Plan
    from paper_2106_09122_gb300.serve import MultiForward
    rng = np.random.default_rng(3)
    plan = Plan(torch.rand(4, n, n, device=DEV), np.linspace(0.0, 3.0, 4), 0.25, N=64, S=0.125, storage="split_bf16")
    x = torch.from_numpy(rng.uniform(0.0, 1.0, (5, 64 * 64)).astype(np.float32))
    out = []
    for units in (1, 40):
        mf = MultiForward([plan], [5], tuning=(0, units, 0))
        mf.x[0].copy_(x)
        mf.count.fill_(5)
        mf.enqueue()
        out.append(mf.y[0].double().cpu())
    assert plan.sync_status() == 0
    assert torch.all((out[0] - out[1]).abs() <= 2e-5 * out[0])


@pytest.mark.parametrize("n,N,n_r,held", [(128, 64, 60, False), (33, 66, 4, True)])
@pytest.mark.parametrize("storage", ["split_bf16", "bf16"])
def test_plan_holds_no_large_tables_and_builds_without_memory_for_them(n, N, n_r, held, storage, monkeypatch):
    """What only the build reads is held where it is small beside A, else given back; when there is
    no memory for it the same A comes out."""
    import ctypes
    from paper_2106_09122_gb300 import Plan, workspace_bytes
    from paper_2106_09122_gb300 import _binding as B
    radii, S = np.linspace(0.0, 5.0, n_r), 8.0 / N
    lib = torch.from_numpy(np.random.default_rng(3).uniform(0.0, 1.0, (n_r, n, n)).astype(np.float32)).to(DEV)
    code = B.SPLIT_BF16 if storage == "split_bf16" else B.BF16
    least, L = ctypes.c_size_t(), B.load()
    B.check(L.psfsim_workspace_min_bytes(n, n_r, N * N, code, ctypes.byref(least)), "workspace_min_bytes")
    full = workspace_bytes(n, n_r, N * N, storage)
    assert full > least.value
    plan = Plan(lib, radii, 0.25, N=N, S=S, storage=storage)
    assert plan.workspace.numel() == (full if held else least.value)
    end = plan.info.scale_offset + 4 * plan.info.ld
    ws, h = torch.zeros(full, dtype=torch.uint8, device=DEV), ctypes.c_void_p()
    B.check(L.psfsim_build(lib.data_ptr(), radii.ctypes.data, n_r, n, 0.25, N, S, code, B.LINEAR, ws.data_ptr(), full, None,
                           ctypes.byref(h)), "psfsim_build")
    torch.cuda.synchronize()
    assert torch.equal(ws[:end], plan.workspace[:end])
    L.psfsim_free(h)
    real, refused = torch.empty, []

    def empty(size, *args, **kw):
        if size == (full if held else full - least.value):
            refused.append(size)
            raise torch.cuda.OutOfMemoryError("no memory")
        return real(size, *args, **kw)

    monkeypatch.setattr(torch, "empty", empty)
    small = Plan(lib, radii, 0.25, N=N, S=S, storage=storage)
    monkeypatch.undo()
    assert refused and small.workspace.numel() == least.value
    assert torch.equal(small.workspace[:end], plan.workspace[:end]) and small.sync_status() == 0


@pytest.mark.parametrize("storage,B", [("split_bf16", 1), ("split_bf16", 9), ("bf16", 3), ("split_bf16_sym", 2)])
@pytest.mark.parametrize("power", [-99, -101, -112, -120, -124])
def test_adjoint_of_very_small_residuals(storage, B, power):
    """Residuals near the bottom of float32's normal range, whose lesser bf16 parts are subnormal: each
    result as exact as for ordinary ones; one residual of ordinary size, one with a few ordinary values
    far from its start, and one of zeros beside them."""
    plan, A, rng = _plan(64, 0.25, 4.0, storage, n=33)
    g = rng.standard_normal((B, 33 * 33)).astype(np.float32)
    g *= np.float32(2.0) ** np.float32(power)
    if B >= 9:
        g[3] = rng.standard_normal(33 * 33)
        g[5, -7:] = 1.0
        g[7] = 0.0
    gx = plan.adjoint(torch.from_numpy(g).to(DEV)).double().cpu().numpy()
    g64 = g.astype(np.float64)
    err = O.bound_relative_error(gx, g64 @ A, np.abs(g64) @ np.abs(A), floor=O.FLT_MIN).max()
    assert err <= ADJOINT_TOL[storage] and plan.sync_status() == 0, err
    assert np.all(gx[:, ~A.any(axis=0)] == 0.0)


@pytest.mark.parametrize("storage,n,N,r_last", [("fp32", 17, 20, 4.0), ("fp32", 40, 24, 30.0), ("fp32", 33, 30, 30.0),
                                                ("fp32", 64, 36, 30.0), ("fp32_sym", 41, 24, 4.0), ("fp32_sym", 32, 48, 30.0),
                                                ("fp32_sym", 24, 52, 30.0), ("fp32_sym", 20, 66, 30.0), ("fp32_sym", 21, 72, 30.0)])
def test_adjoint_of_few_columns(storage, n, N, r_last):
    """Passes of 8, 4 and 2 residuals on few columns (up to 608 and 1216 of them on 152 SMs, between and
    above), the remainders that take the batched form, odd images, residuals at any 4-byte address; a
    dense grid with and without dead columns, and infinities."""
    plan, A, rng = _plan(N, 8.0 / N, r_last, storage, n=n)
    for B in (1, 2, 3, 4, 7, 8, 9, 10, 12, 15, 16, 18):
        big = torch.from_numpy(rng.standard_normal(B * n * n + 1).astype(np.float32)).to(DEV)
        for shift in (0, 1):
            g = big[shift:shift + B * n * n].view(B, n * n)
            gx = plan.adjoint(g).double().cpu().numpy()
            g64 = g.double().cpu().numpy()
            err = O.bound_relative_error(gx, g64 @ A, np.abs(g64) @ np.abs(A), floor=O.FLT_MIN).max()
            assert err <= 1e-5 and plan.sync_status() == 0, (B, shift, err)
            assert np.all(gx[:, ~A.any(axis=0)] == 0.0)
    if storage == "fp32":
        g = big[:8 * n * n].view(8, n * n).clone()
        g[5, 3] = float("inf")
        gx = plan.adjoint(g).cpu().numpy()
        assert np.isfinite(gx[[0, 1, 2, 3, 4, 6, 7]]).all() and not np.isfinite(gx[5][A[3] == 0.0]).any()


@pytest.mark.parametrize("storage", ["split_bf16", "bf16"])
@pytest.mark.parametrize("n,N,r_last", [(17, 91, 30.0), (16, 128, 12.0), (33, 96, 30.0), (24, 90, 30.0)])
def test_adjoint_of_one_residual_where_nearly_all_columns_are_read(storage, n, N, r_last):
    """One residual on CUDA cores (from 8192 columns on) and, below, on the tensor cores: odd images and
    grids, column counts off the 8 of a thread; the same residual in a batch; infinities; small values."""
    plan, A, rng = _plan(N, 8.0 / N, r_last, storage, n=n)
    g = rng.standard_normal((2, n * n)).astype(np.float32)
    for x in (g, np.float32(2.0 ** -120) * g):
        x64 = x.astype(np.float64)
        one = plan.adjoint(torch.from_numpy(x[0]).to(DEV)).double().cpu().numpy()
        two = plan.adjoint(torch.from_numpy(x).to(DEV)).double().cpu().numpy()
        for y, r in ((one[None], x64[:1]), (two, x64)):
            err = O.bound_relative_error(y, r @ A, np.abs(r) @ np.abs(A), floor=O.FLT_MIN).max()
            assert err <= ADJOINT_TOL[storage] and plan.sync_status() == 0, err
        assert np.all(one[~A.any(axis=0)] == 0.0)
    g[0, 5] = -np.inf
    y = plan.adjoint(torch.from_numpy(g[0]).to(DEV)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = np.where(A[5] == 0.0, np.nan, -np.inf)
    assert np.array_equal(y, want.astype(np.float32), equal_nan=True)
