"""The float64 nonlocal term of hpsi_apply_batch on both sides of the lines between the tiles over all items and the digit
products item by item: 16 and 17 projectors, and 6e6 multiply-adds an item."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
SMALL, LARGE = (8.0, 8.0), (14.0, 12.0)   # cell edge and cutoff: 515 and 5449 plane waves


def _setup(items, precision):
    """items: (cell, projectors, bands); random projectors and a D that couples them."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    lats, ecuts, ffts, vrs, betas, ds, xs = [], [], [], [], [], [], []
    for i, ((a, ecut), nproj, nb) in enumerate(items):
        rng = np.random.default_rng(i)
        lat = np.diag([a, a, a])
        m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
        n = workloads.cubic_box(a, ecut)
        lats.append(lat)
        ecuts.append(ecut)
        ffts.append((n, n, n))
        vrs.append(rng.standard_normal((n, n, n)))
        betas.append((rng.standard_normal((nproj, len(m))) + 1j * rng.standard_normal((nproj, len(m)))) / np.sqrt(len(m)))
        d = rng.standard_normal((nproj, nproj)) + 1j * rng.standard_normal((nproj, nproj))
        ds.append((d + d.conj().T) / 2)
        xs.append(torch.from_numpy(workloads.random_block(len(m), nb, i)).cuda())
    ctx = B.hpsi_setup_cells(lats, ecuts, ffts, vrs, betas, ds, precision, torch.cuda.current_stream().cuda_stream)
    return ctx, xs, betas, ds


def _batch(ctx, xs, ys):
    from paper_0906_2569_gb300 import binding as B
    for y in ys:
        y.fill_(float("nan"))
    B.hpsi_apply_batch(ctx, list(range(len(xs))), xs, ys)
    B.hpsi_sync(ctx)
    return [y.cpu().numpy() for y in ys]


MANY = [(SMALL, p, nb) for p, nb in [(16, 5), (17, 5), (24, 31), (33, 8), (1, 1), (64, 24), (20, 9), (48, 2)]]


@pytest.mark.parametrize("precision", [0, 1])
def test_small_items_share_one_launch(lib, precision):
    from paper_0906_2569_gb300 import binding as B
    ctx, xs, _, _ = _setup(MANY, precision)
    ys = [x.clone() for x in xs]
    B.hpsi_kernel_stats(ctx, -1, reset=True)
    _batch(ctx, xs, ys)
    for k in ("calbec", "addvus"):
        assert B.hpsi_kernel_stats(ctx, B.KERNELS.index(k))[0] == 1
    ctx.close()


@pytest.mark.parametrize("items", [MANY, [(LARGE, 40, 33)] + MANY[:3] + [(LARGE, 17, 60)], [(SMALL, 90, 17), (SMALL, 20, 40)],
                                   [(SMALL, 12, 4), (SMALL, 16, 33)]])
def test_batch_against_single_calls(lib, items):
    """Float64: to rounding of the sums (both sides add 2 npw and 2 P products, up to sqrt(terms) 2^-53 each, and the two
    terms of H), and the same bits where both take the same form; the replay and the persistent launch give the same
    bits as the first call."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    ctx, xs, betas, ds = _setup(items, B.HPSI_FP64)
    ys = [torch.empty_like(x) for x in xs]
    first = _batch(ctx, xs, ys)
    again = _batch(ctx, xs, ys)
    B.hpsi_set_option(ctx, B.HPSI_OPT_PERSISTENT, 1)
    pers = _batch(ctx, xs, ys)
    for i, (x, (_, nproj, nb)) in enumerate(zip(xs, items)):
        y = torch.full_like(x, float("nan"))
        B.hpsi_apply(ctx, i, x, y)
        B.hpsi_sync(ctx)
        y = y.cpu().numpy()
        assert np.array_equal(first[i], again[i]) and np.array_equal(first[i], pers[i])
        npw = x.shape[1]
        if nproj <= 16 or nproj * npw * nb >= 6e6:
            assert np.array_equal(first[i], y)
        nl = (x.cpu().numpy() @ betas[i].conj().T) @ ds[i].T @ betas[i]
        for b in range(nb):
            tol = 4 * (np.sqrt(2.0 * npw) + np.sqrt(2.0 * nproj) + 4) * 2.0 ** -53 * np.linalg.norm(nl[b])
            assert np.linalg.norm(first[i][b] - y[b]) <= tol + 4 * 2.0 ** -53 * np.linalg.norm(y[b])
    ctx.close()


def test_mixed_batch_on_both_sides(lib):
    """Mixed context, every item up to 64 projectors: the float64 nonlocal term of the batch, in either form, within float32
    accuracy of the single calls; the replay gives the same bits."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    ctx, xs, _, _ = _setup(MANY[:4] + [(LARGE, 40, 33)], B.HPSI_MIXED)
    ys = [torch.empty_like(x) for x in xs]
    first = _batch(ctx, xs, ys)
    again = _batch(ctx, xs, ys)
    for i, x in enumerate(xs):
        y = torch.full_like(x, float("nan"))
        B.hpsi_apply(ctx, i, x, y)
        B.hpsi_sync(ctx)
        y = y.cpu().numpy()
        assert np.array_equal(first[i], again[i])
        assert np.linalg.norm(first[i] - y) <= 1e-5 * np.linalg.norm(y)
    ctx.close()
