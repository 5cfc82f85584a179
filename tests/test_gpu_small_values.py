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


@pytest.mark.parametrize("e", [0, 90, 118])
def test_mixed_gamma_nonlocal_of_large_bands(lib, e):
    """Bands of up to 2^118: the nonlocal term of the Gamma form alone (V = 0) stays in float32's range and scales with the
    band (all its operands and sums are floating-point numbers of eight exponent bits)."""
    lat, ecut, n = np.diag([8.0, 8.0, 8.0]), 8.0, 20
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
    beta = workloads.beta(lat, np.random.default_rng(1).random((5, 3)) @ lat, np.zeros(3), m)
    psi = workloads.random_block(len(m), 3, 3)[:, len(m) // 2:].copy()
    psi[:, 0] = psi[:, 0].real
    args = (lat, ecut, (n, n, n), np.zeros((n, n, n)), [beta], workloads.dmat(5), B.HPSI_MIXED)
    one, large = _apply(*args, psi, True), _apply(*args, psi * 2.0 ** e, True) * 2.0 ** -e
    assert np.linalg.norm(large - one) <= 1e-6 * np.linalg.norm(one)


def _float64_case(gamma, nproj=20):
    from paper_0906_2569_gb300 import binding as B
    lat, ecut, n = np.diag([8.0, 8.0, 8.0]), 8.0, 20
    m = B.hpsi_gsphere(lat, ecut, np.zeros(3))
    rng = np.random.default_rng(1)
    atoms = rng.random((nproj // 4, 3)) @ lat
    beta = workloads.beta(lat, atoms, np.zeros(3), m)
    v = rng.uniform(-1.0, 1.0, size=(n, n, n))
    psi = workloads.random_block(len(m), 3, 3)
    if gamma:
        psi = psi[:, len(m) // 2:].copy()
        psi[:, 0] = psi[:, 0].real
    return lat, ecut, (n, n, n), v, [beta], workloads.dmat(nproj // 4), B.HPSI_FP64, psi


def _ldexp(x, e):
    return np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e)


@pytest.mark.parametrize("gamma", [False, True])
@pytest.mark.parametrize("e", [-960, -990, -1010, 960])
def test_float64_scales_exactly(lib, gamma, e):
    """A power of two on normal numbers: every step of H scales exactly, so only results below 2^-1022 are rounded (at
    2^-1074, in the local, kinetic and nonlocal term and their two sums, and in the two bands of a Gamma pair)."""
    case = _float64_case(gamma)
    psi = case[-1]
    one, small = _apply(*case, gamma), _apply(*case[:-1], _ldexp(psi, e), gamma)
    d = small - _ldexp(one, e)
    assert max(np.abs(d.real).max(), np.abs(d.imag).max()) <= (16 * 2.0 ** -1074 if e < 0 else 0.0)


@pytest.mark.parametrize("gamma", [False, True])
def test_float64_subnormal_bands(lib, gamma):
    """Coefficients of about 2^-1060, kept to 2^-1074: H of them, within the roundings at 2^-1074 named above and those of
    <beta|psi>, which 20 projectors of D and beta up to 4 take along."""
    case = _float64_case(gamma)
    x = _ldexp(case[-1], -1060)
    up = _apply(*case[:-1], _ldexp(x, 1060), gamma)
    d = _apply(*case[:-1], x, gamma) - _ldexp(up, -1060)
    assert np.abs(up).max() > 2.0   # 2^14 steps of 2^-1074
    assert max(np.abs(d.real).max(), np.abs(d.imag).max()) <= (16 + 20 * 4) * 2.0 ** -1074


def test_float64_subnormal_potential_and_projectors(lib):
    """V and the projectors near 2^-1060 on a band that is G = 0 alone, where the kinetic term vanishes."""
    lat, ecut, fft, v, beta, d, prec, psi = _float64_case(False, 20)
    npw = psi.shape[1]
    one = np.zeros((1, npw), dtype=complex)
    one[0, npw // 2] = 2.0 ** 30
    tiny = _ldexp(v, -1060).real
    y = _apply(lat, ecut, fft, tiny, None, None, prec, one)
    want = np.ldexp(tiny, 1060).mean() * 2.0 ** 30
    assert abs(np.ldexp(y[0, npw // 2].real, 1060) - want) <= 1e-3 * abs(want)
    # <beta|psi> = 2^30 conj(beta(0)) 2^-1060 is subnormal-free; the sum over p runs with normal projectors in the second term
    b = np.zeros((20, npw), dtype=complex)
    b[:, npw // 2] = np.ldexp(np.arange(1.0, 21.0), -1060)
    one[0, npw // 2] = 2.0 ** 1000
    y = _apply(lat, ecut, fft, 0 * v, [b], np.diag(np.full(20, 2.0 ** 1000 + 0j)), prec, one)
    want = (np.arange(1.0, 21.0) ** 2).sum() * 2.0 ** (1000 + 1000 - 1060 - 1060)
    assert abs(y[0, npw // 2] - want) <= 2.0 ** -40 * want
