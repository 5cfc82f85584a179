"""Bands and operators of very small values: what a power of two does to H|psi> in a mixed context, float32 values below
float32's normal range."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _apply(lat, ecut, fft, v, beta, d, precision, x, gamma=False):
    import torch
    from paper_0906_2569_gb300 import binding as B
    ctx = B.hpsi_setup(lat, ecut, [np.zeros(3)], fft, v, beta, d, precision, torch.cuda.current_stream().cuda_stream)
    B.hpsi_set_option(ctx, B.HPSI_OPT_AUTOTUNE, 0)
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.full_like(xd, float("nan"))
    (B.hpsi_apply_gamma if gamma else B.hpsi_apply)(ctx, 0, xd, y)
    B.hpsi_sync(ctx)
    ctx.close()
    return y.cpu().numpy()


@pytest.mark.parametrize("gamma", [False, True])
def test_mixed_local_term_of_small_bands(lib, gamma):
    """Coefficients of 2^-118 (3e-36) are normal float32 numbers, and so are all sums over them: the local term is as
    accurate as that of coefficients of the order of 1 (other roundings, the same size: at most twice the error)."""
    import oracle
    from paper_0906_2569_gb300 import binding as B
    n, a, ecut = 100, 20.0, 8.0
    lat = np.diag([a, a, a])
    m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
    npw = len(m)
    psi = workloads.random_block(npw, 2, 3)
    if gamma:
        psi = psi[:, npw // 2:].copy()
        psi[:, 0] = psi[:, 0].real
    full = np.concatenate([psi[:, 1:][:, ::-1].conj(), psi], axis=1) if gamma else psi
    v = np.random.default_rng(0).uniform(-1.0, 1.0, size=(n, n, n))
    ref = oracle.hamiltonian.local_term(v, m, (n, n, n), full)[:, -psi.shape[1]:]
    kin = _apply(lat, ecut, (n, n, n), np.zeros_like(v), None, None, B.HPSI_MIXED, psi, gamma)
    err = []
    for s in (1.0, 2.0 ** -118):
        y = _apply(lat, ecut, (n, n, n), v, None, None, B.HPSI_MIXED, psi * s, gamma) / s
        err.append(np.linalg.norm(y - kin - ref) / np.linalg.norm(ref))
    assert err[0] < 1e-6 and err[1] <= 2.0 * err[0]
