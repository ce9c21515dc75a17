"""Scratch sizes against what the launches of a call take, on the host: the size that a caller asks
for is never below the partial images and split scenes that the product then writes."""
import ctypes

import numpy as np
import pytest

from paper_2106_09122_gb300 import _binding as B

STORAGES = {"split_bf16": B.SPLIT_BF16, "bf16": B.BF16, "split_bf16_sym": B.SPLIT_BF16_SYM}


def _scratch(n, N, storage, batch, r_last=12.0, field=32.0, num_sms=152, adjoint=0):
    radii = np.linspace(0.0, r_last, 5)
    reported, taken, run = ctypes.c_size_t(), ctypes.c_size_t(), ctypes.c_int()
    B.check(B.load().psfsim_debug_scratch(radii.ctypes.data, 5, n, N, field / N, STORAGES[storage], num_sms, adjoint,
                                          batch, ctypes.byref(reported), ctypes.byref(taken), ctypes.byref(run)),
            "psfsim_debug_scratch")
    return reported.value, taken.value, run.value


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n", [16, 24, 64, 128, 160, 256])
def test_forward_scratch_holds_every_launch(storage, n):
    for N in (32, 60, 64, 96, 128, 200, 256):
        for num_sms in (148, 152):
            for batch in (1, 2, 3, 5, 10, 16, 17, 20, 21, 33, 64, 80, 81, 130, 320, 321, 336, 1280, 1281, 1340, 2480):
                reported, taken, _ = _scratch(n, N, storage, batch, num_sms=num_sms)
                assert reported >= taken, (N, num_sms, batch)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n", [16, 18, 22, 24, 64, 160])
def test_adjoint_scratch_holds_every_launch(storage, n):
    """More than 1280 residuals (320 on compact storage) take several launches, of which the last
    may split k further than the first.  All columns live, or 44 % of them."""
    for N in (20, 32, 60, 64, 66, 100, 160):
        for field, num_sms in ((32.0, 152), (32.0, 148), (16.0, 152)):
            for batch in (1, 5, 20, 21, 80, 81, 320, 321, 350, 560, 600, 640, 1280, 1281, 1300, 1400, 2240, 2480, 2560):
                reported, taken, _ = _scratch(n, N, storage, batch, field=field, num_sms=num_sms, adjoint=1)
                assert reported >= taken, (N, field, num_sms, batch)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n,N", [(64, 64), (16, 60), (24, 100), (100, 86), (128, 32), (160, 64), (256, 128)])
def test_scratch_for_a_batch_serves_every_smaller_one(storage, n, N):
    for adjoint in (0, 1):
        most = 0
        for batch in [*range(1, 100), 128, 129, 160, 161, 200, 256, 257, 320, 321, 400, 1280, 1281, 2480]:
            reported, taken, _ = _scratch(n, N, storage, batch, adjoint=adjoint)
            assert reported >= max(most, taken), (adjoint, batch)
            most = reported


@pytest.mark.parametrize("storage", ["split_bf16", "split_bf16_sym"])
@pytest.mark.parametrize("n,N", [(64, 64), (128, 128), (256, 128), (256, 256), (400, 64)])
def test_adjoint_of_split_storage_adds_short_runs_whatever_the_batch(storage, n, N):
    """At most 160 k-tiles of 64 image rows in one FP32 chain, with one job or several."""
    for batch in (1, 8, 16, 20, 21, 64, 80, 81, 100, 160, 161, 320, 321, 1280, 1281):
        assert _scratch(n, N, storage, batch, adjoint=1)[2] <= 160, batch


def _guarded(plan, product, x, need):
    """The product with a scratch of exactly `need` bytes, and whether the 64 KiB after it are as they were."""
    import torch
    guard = 1 << 16
    buf = torch.full((need + guard,), 0x5A, dtype=torch.uint8, device=x.device)
    out = product(x, scratch=buf[:need])
    assert plan.sync_status() == 0
    return out, bool(torch.all(buf[need:] == 0x5A))


@pytest.mark.gpu
@pytest.mark.parametrize("n,N,batch", [(64, 32, 1), (64, 32, 16), (128, 32, 5), (160, 64, 10), (24, 96, 17)])
def test_compact_forward_stays_inside_its_scratch(n, N, batch):
    """Few columns, so that several splits are worth their partial images, which compact storage
    always has.  Sums of products that are not negative: both within 1e-5 of the true ones."""
    import torch
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(n + N)
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (5, n, n)).astype(np.float32)).cuda()
    radii, S = np.linspace(0.0, 12.0, 5), 32.0 / N
    x = torch.from_numpy(rng.uniform(0.0, 1.0, (batch, N * N)).astype(np.float32)).cuda()
    split = Plan(lib, radii, 0.25, N=N, S=S, storage="split_bf16_sym")
    y, clean = _guarded(split, split.forward, x, split.forward_scratch_bytes(batch))
    assert clean
    ref = Plan(lib, radii, 0.25, N=N, S=S, storage="fp32_sym").forward(x)
    assert torch.all((y.double() - ref.double()).abs() <= 2e-5 * ref.double())


@pytest.mark.gpu
@pytest.mark.parametrize("n,N,storage,batch", [(16, 60, "split_bf16", 1281), (16, 60, "bf16", 2480),
                                               (16, 60, "split_bf16", 2480), (16, 60, "split_bf16_sym", 321),
                                               (24, 100, "split_bf16_sym", 600)])
def test_adjoint_of_several_launches_stays_inside_its_scratch(n, N, storage, batch):
    """Residuals that are not negative: sums without cancellation, within 1e-5 of the true ones
    (BF16: and 2^-8 of them)."""
    import torch
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(n + N)
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (5, n, n)).astype(np.float32)).cuda()
    radii, S = np.linspace(0.0, 12.0, 5), 16.0 / N
    g = torch.from_numpy(rng.uniform(0.0, 1.0, (batch, n * n)).astype(np.float32)).cuda()
    split = Plan(lib, radii, 0.25, N=N, S=S, storage=storage)
    gx, clean = _guarded(split, split.adjoint, g, split.adjoint_scratch_bytes(batch))
    assert clean
    ref = Plan(lib, radii, 0.25, N=N, S=S).adjoint(g).double()
    tol = 2e-5 + (2.0 ** -8 if storage == "bf16" else 0.0)
    assert torch.all((gx.double() - ref).abs() <= tol * ref)


@pytest.mark.gpu
@pytest.mark.parametrize("storage,n,N", [("split_bf16", 64, 64), ("bf16", 100, 86)])
def test_multi_forward_scratch_of_one_job_serves_smaller_capacities(storage, n, N):
    import torch
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(n)
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (5, n, n)).astype(np.float32)).cuda()
    plan = Plan(lib, np.linspace(0.0, 12.0, 5), 0.25, N=N, S=32.0 / N, storage=storage)
    x = torch.from_numpy(rng.uniform(0.0, 1.0, (80, N * N)).astype(np.float32)).cuda()
    y = torch.empty((80, n * n), device="cuda")
    L, nb = B.load(), ctypes.c_size_t()

    def job(cap):
        return (B.Job * 1)(B.Job(plan.handle, x.data_ptr(), y.data_ptr(), cap, None))

    B.check(L.psfsim_forward_multi_scratch_bytes(job(80), 1, None, ctypes.byref(nb)), "scratch")
    scr = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    ref = plan.forward(x)
    most = 0
    for cap in range(1, 81):
        B.check(L.psfsim_forward_multi_scratch_bytes(job(cap), 1, None, ctypes.byref(nb)), "scratch")
        assert nb.value >= most
        most = nb.value
        B.check(L.psfsim_forward_multi(job(cap), 1, None, scr.data_ptr(), scr.numel(),
                                       torch.cuda.current_stream().cuda_stream), "psfsim_forward_multi")
        tol = 2e-5 * ref[:cap]  # both sums of products that are not negative, split differently
        assert torch.all((y[:cap] - ref[:cap]).abs() <= tol)
    assert plan.sync_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("batch", [1, 17, 90, 350, 1300])
def test_scratch_below_what_a_call_takes_is_refused_before_anything_runs(storage, batch):
    import torch
    from paper_2106_09122_gb300 import Plan
    n, N = 16, 24
    rng = np.random.default_rng(5)
    lib = torch.from_numpy(rng.uniform(0.0, 1.0, (5, n, n)).astype(np.float32)).cuda()
    L, st = B.load(), torch.cuda.current_stream().cuda_stream
    for radii in (np.linspace(0.0, 12.0, 5), np.linspace(0.0, 0.1, 5)):  # the second: no column at all
        plan = Plan(lib, radii, 0.25, N=N, S=1.0, storage=storage)
        x, g = torch.ones(batch, N * N, device="cuda"), torch.ones(batch, n * n, device="cuda")
        for call, a, out, nbytes in ((L.psfsim_forward, x, torch.full_like(g, 7.0), plan.forward_scratch_bytes(batch)),
                                     (L.psfsim_adjoint, g, torch.full_like(x, 7.0), plan.adjoint_scratch_bytes(batch))):
            scr = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

            def run(size, ptr=scr.data_ptr()):
                return call(plan.handle, a.data_ptr(), batch, out.data_ptr(), ptr, size, st)

            assert run(0) == B.ERR_WORKSPACE and run(255) == B.ERR_WORKSPACE and run(nbytes, None) == B.ERR_WORKSPACE
            assert run(nbytes, scr.data_ptr() + 16) == B.ERR_WORKSPACE
            low, high = 255, nbytes  # the least that is accepted; everything below is refused and leaves the output alone
            while high - low > 1:
                mid = (low + high) // 2
                torch.cuda.synchronize()
                before = out.clone()
                rc = run(mid)
                assert rc in (B.OK, B.ERR_WORKSPACE)
                torch.cuda.synchronize()
                assert rc == B.OK or torch.equal(out, before)
                low, high = (low, mid) if rc == B.OK else (mid, high)
            assert run(high) == B.OK and plan.sync_status() == 0
