"""hpsi_apply_gamma in a mixed context returns float64: the nonlocal term's float32 partial sums (one per 512 projectors) are
added to more than float32 accuracy, as in the complex form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LAT, ECUT, FFT = np.diag([8.0, 8.0, 8.0]), 8.0, (20, 20, 20)


def test_cancelling_partial_sums(lib):
    """Three groups of 512 projectors, each with one on G = 0 alone, and D = 2^24, 1, -2^24: every product and partial sum is
    exact, and their sum is 1 only if the 1 survives beside 2^24."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(LAT, ECUT, np.zeros(3))
    npw = len(m)
    P = 3 * 512
    beta = np.zeros((P, npw), dtype=complex)
    beta[:, npw // 2] = 1.0
    d = np.zeros((P, P), dtype=complex)
    for g, v in enumerate((2.0 ** 24, 1.0, -2.0 ** 24)):
        d[512 * g + 3, 512 * g + 3] = v
    ctx = B.hpsi_setup(LAT, ECUT, [np.zeros(3)], FFT, np.zeros(FFT), [beta], d, B.HPSI_MIXED,
                       torch.cuda.current_stream().cuda_stream)
    x = torch.zeros(3, (npw + 1) // 2, dtype=torch.complex128, device="cuda")
    x[:, 0] = torch.tensor([1.0, -0.5, 3.0])
    y = torch.full_like(x, float("nan"))
    B.hpsi_apply_gamma(ctx, 0, x, y)
    B.hpsi_sync(ctx)
    ctx.close()
    # G = 0 has no kinetic term, and V = 0
    assert np.array_equal(y.cpu().numpy(), x.cpu().numpy())
