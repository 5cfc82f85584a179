"""The digit planes of the projectors (four times the projectors' memory) are a cache: a call that finds the device's memory
taken goes on without them, and other workspaces can have their memory back."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
MB = 1 << 20
LAT, ECUT, P = np.diag([14.0, 14.0, 14.0]), 12.0, 256   # 5449 plane waves: planes of 2 x 45 MB


def _fill(leave):
    """Device memory taken until about `leave` bytes are free."""
    import torch
    held = []
    torch.cuda.empty_cache()
    for _ in range(40):
        want = torch.cuda.mem_get_info()[0] - leave
        if want < 2 * MB:
            break
        try:
            held.append(torch.empty(want // (2 * MB) * (2 * MB), dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            leave += 2 * MB
    return held


def _context(gamma):
    import torch
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(LAT, ECUT, np.zeros(3))
    n = workloads.cubic_box(14.0, ECUT)
    rng = np.random.default_rng(0)
    beta = workloads.beta(LAT, rng.random((P // 4, 3)) @ LAT, np.zeros(3), m)
    v = rng.standard_normal((n, n, n))
    make = lambda: B.hpsi_setup(LAT, ECUT, [np.zeros(3)], (n, n, n), v, [beta], workloads.dmat(P // 4), B.HPSI_FP64,
                                torch.cuda.current_stream().cuda_stream)
    x = torch.from_numpy(workloads.random_block(len(m), 160, 1)).cuda()
    if gamma:
        x = x[:, len(m) // 2:].contiguous()
        x[:, 0].imag.zero_()
    return make, x, B.hpsi_apply_gamma if gamma else B.hpsi_apply


def _reference(make, x, apply):
    """H x with all the memory there is; the kernels without the planes are loaded too (a module needs memory)."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    ctx = make()
    ref = torch.empty_like(x)
    apply(ctx, 0, x, ref)
    if apply is B.hpsi_apply:
        B.hpsi_apply_noalloc(ctx, 0, x[:2], torch.empty_like(x[:2]))
        B.hpsi_apply_noalloc(ctx, 0, x, torch.empty_like(x))
    B.hpsi_sync(ctx)
    ctx.close()
    return ref


def _same(y, ref, npw):
    # both sides' sums of 2 npw and 2 P products, up to sqrt(terms) 2^-53 each, on a norm of D beta psi below that of H psi
    tol = 4 * (np.sqrt(2.0 * npw) + np.sqrt(2.0 * P) + 4) * 2.0 ** -53
    return float((y - ref).abs().square().sum().sqrt() / ref.abs().square().sum().sqrt()) < tol


def test_workspaces_get_the_planes_memory_back(lib):
    import torch
    from paper_0906_2569_gb300 import binding as B
    make, x, apply = _context(False)
    ref = _reference(make, x, apply)
    y = torch.empty_like(x)
    ctx = make()
    apply(ctx, 0, x[:2], y[:2])   # makes the planes and small workspaces
    B.hpsi_sync(ctx)
    held = _fill(20 * MB)
    try:
        apply(ctx, 0, x, y)       # the stick rows alone are 2 x 25 MB
        B.hpsi_sync(ctx)
    finally:
        del held
        torch.cuda.empty_cache()
    assert _same(y, ref, x.shape[1])
    apply(ctx, 0, x, y)
    B.hpsi_sync(ctx)
    assert _same(y, ref, x.shape[1])
    ctx.close()


def test_no_half_of_the_planes_is_kept(lib):
    """Room for one set of planes but not for both: the call goes on without, and holds none."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    make, x, apply = _context(False)
    ref = _reference(make, x, apply)
    y = torch.empty_like(x[:16])
    ctx = make()
    held = _fill(70 * MB)
    try:
        before = torch.cuda.mem_get_info()[0]
        apply(ctx, 0, x[:16], y)
        B.hpsi_sync(ctx)
        after = torch.cuda.mem_get_info()[0]
    finally:
        del held
        torch.cuda.empty_cache()
    assert _same(y, ref[:16], x.shape[1])
    assert before - after < 40 * MB   # 16 bands' workspaces, no set of 45 MB
    ctx.close()


def test_gamma_goes_on_without_planes(lib):
    import torch
    from paper_0906_2569_gb300 import binding as B
    make, x, apply = _context(True)
    ref = _reference(make, x, apply)
    # the kernels of the other form
    small = torch.empty_like(x)
    ctx = make()
    apply(ctx, 0, x[:1], small[:1])
    B.hpsi_sync(ctx)
    held = _fill(40 * MB)   # the call needs about 70, the planes are 45
    try:
        apply(ctx, 0, x, small)
        B.hpsi_sync(ctx)
    finally:
        del held
        torch.cuda.empty_cache()
    assert _same(small, ref, 2 * x.shape[1])
    ctx.close()
