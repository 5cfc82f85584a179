"""The float32 local term on average: <psi|V|psi> of mixed contexts.  The roundings of single values average out over a band;
those of the transforms' constants do not, unless they are corrected for (up to 1.8e-7 of <psi|V|psi> on an 81^3 box).

Tolerance: what the correction leaves per axis differs from index to index by 2.2e-8 at most (standard deviation over the
box's indices, from the constants alone); three axes, averaged over at least 11 indices each: 3 x 2.2e-8 / sqrt(11) = 2e-8.
The float32 noise of single values, 4e-7 over the square root of the thousands of coefficients, and V's own rounding,
3e-8 over that of the grid points, come below 1e-8."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mmax", [(25, 6), (27, 6), (36, 8), (50, 12), (54, 12), (64, 15), (81, 19), (100, 12), (108, 12)])
@pytest.mark.parametrize("gamma", [False, True])
def test_mean_of_the_local_term(lib, n, mmax, gamma):
    import torch
    from paper_0906_2569_gb300 import binding as B
    ecut = 8.0
    a = 2.0 * np.pi * (mmax + 0.3) / np.sqrt(2.0 * ecut)
    lat = np.diag([a, a, a])
    m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
    npw = len(m)
    rng = np.random.default_rng(n)
    v = rng.uniform(0.5, 1.5, size=(n, n, n))
    nb = max(2, 20000 // npw)
    psi = workloads.random_block(npw, nb, 1)
    if gamma:
        psi = (psi + psi[:, ::-1].conj()) / 2.0
    x = torch.from_numpy(np.ascontiguousarray(psi[:, npw // 2:] if gamma else psi)).cuda()
    ys = []
    for pot in (v, np.zeros_like(v)):   # V = 0 leaves the kinetic term
        ctx = B.hpsi_setup(lat, ecut, [np.zeros(3)], (n, n, n), pot, None, None, B.HPSI_MIXED,
                           torch.cuda.current_stream().cuda_stream)
        y = torch.empty_like(x)
        (B.hpsi_apply_gamma if gamma else B.hpsi_apply)(ctx, 0, x, y)
        B.hpsi_sync(ctx)
        ctx.close()
        ys.append(y.cpu().numpy())
    got = ys[0] - ys[1]
    if gamma:
        got = np.concatenate([got[:, 1:][:, ::-1].conj(), got], axis=1)
    box = np.zeros((nb, n, n, n), dtype=complex)
    box[:, m[:, 0] % n, m[:, 1] % n, m[:, 2] % n] = psi
    r = np.fft.ifftn(box, axes=(1, 2, 3), norm="forward")
    ref = (np.abs(r) ** 2 * v).sum() / n ** 3
    assert abs((psi.conj() * got).sum().real / ref - 1.0) < 3e-8
