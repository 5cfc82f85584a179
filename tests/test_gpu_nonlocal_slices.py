"""The float64 nonlocal term as exact digit products on the tensor cores (csrc/nonlocal_slices.cu): tile and K remainders,
digits at their extremes (where an inexact accumulation would show at once), scales, zeros and non-finite values."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
FFT = (32, 32, 32)
LAT = np.diag([10.0, 10.0, 10.0])


def _miller():
    from paper_0906_2569_gb300 import binding as B
    return B.hpsi_gsphere(LAT, 10.0, np.zeros(3))


def _apply(beta, d, psi, gamma=False):
    import torch
    from paper_0906_2569_gb300 import binding as B
    ctx = B.hpsi_setup(LAT, 10.0, [np.zeros(3)], FFT, np.zeros(FFT), [beta], d, B.HPSI_FP64,
                       torch.cuda.current_stream().cuda_stream)
    x = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    y = torch.full_like(x, float("nan"))
    (B.hpsi_apply_gamma if gamma else B.hpsi_apply)(ctx, 0, x, y)
    B.hpsi_sync(ctx)
    ctx.close()
    return y.cpu().numpy()


def _tol(npw, nproj):
    """The oracle's own float64 sums of 2 npw and 2 nproj terms round by up to sqrt(terms) 2^-53 each (random signs)."""
    return 2.0 * (np.sqrt(2.0 * npw) + np.sqrt(2.0 * nproj) + 4.0) * 2.0 ** -53


@pytest.mark.parametrize("nproj,nb", [(17, 1), (24, 31), (127, 32), (128, 33), (129, 5), (260, 70)])
def test_tiles_against_oracle(lib, nproj, nb):
    m = _miller()
    rng = np.random.default_rng(nproj)
    beta = (rng.standard_normal((nproj, len(m))) + 1j * rng.standard_normal((nproj, len(m)))) / np.sqrt(len(m))
    d = rng.standard_normal((nproj, nproj)) + 1j * rng.standard_normal((nproj, nproj))
    d = (d + d.conj().T) / 2
    psi = workloads.random_block(len(m), nb, 7)
    psi *= 10.0 ** rng.uniform(-200, 200, size=(nb, 1))
    y = _apply(beta, d, psi)
    kin = oracle.gsphere.kinetic(LAT, np.zeros(3), m)
    for b in range(nb):
        s = np.max(np.abs(psi[b]))
        nl = oracle.hamiltonian.nonlocal_term(beta, d, psi[b:b + 1] / s)[0]
        ref = nl + kin * (psi[b] / s)
        # one rounding more where the two terms are added, and the diagonal's own rounding (twice 2^-53 of it)
        err = np.linalg.norm(y[b] / s - ref)
        assert err < _tol(len(m), nproj) * np.linalg.norm(nl) + 4 * 2.0 ** -53 * np.linalg.norm(kin * psi[b] / s)


@pytest.mark.parametrize("nproj,nb", [(1, 1), (8, 3), (130, 65)])
def test_gamma_tiles_against_complex(lib, nproj, nb):
    m = _miller()
    npw = len(m)
    rng = np.random.default_rng(nproj)
    nat = max(1, nproj // 4)
    beta = workloads.beta(LAT, rng.random((nat, 3)) @ LAT, np.zeros(3), m)[:nproj]
    d = workloads.dmat(nat)[:len(beta), :len(beta)]
    half = workloads.random_block(npw, nb, 3)[:, npw // 2:].copy()
    half[:, 0] = half[:, 0].real
    full = np.concatenate([half[:, 1:][:, ::-1].conj(), half], axis=1)
    y = _apply(beta, d, half, gamma=True)
    none = np.zeros(FFT)
    ref = oracle.hamiltonian.hpsi(LAT, np.zeros(3), m, FFT, none, beta, d, full)[:, npw // 2:]
    nl = oracle.hamiltonian.nonlocal_term(beta, d, full)
    assert np.linalg.norm(y - ref) < _tol(npw, nproj) * np.linalg.norm(nl) + 8 * 2.0 ** -53 * np.linalg.norm(ref)


@pytest.mark.parametrize("pattern", [0x7F7F7F7F7F7F7F, 0x80808080808080, 0x40FFFFFFFFFFFF, 0x55555555555555])
def test_extreme_digits_are_summed_exactly(lib, pattern):
    """Constant projectors and bands whose digits are all near +127 or -128: each accumulator reaches its limit of
    2^24 with equal signs, and the result must still be the correctly scaled integer."""
    m = _miller()
    npw, P = len(m), 17
    x = float(pattern >> 3)           # 53 significant bits at most
    x = x / 2.0 ** 53
    beta = np.full((P, npw), x, dtype=complex)
    psi = np.full((3, npw), -x, dtype=complex)
    psi[1] = x * 1j
    y = _apply(beta, np.eye(P), psi)
    kin = np.array([Fraction(float(v)) for v in oracle.gsphere.kinetic(LAT, np.zeros(3), m)])
    f = Fraction(x)
    w = float(f * f * npw)            # <beta|psi> as the nearest float64
    for b, (vr, vi) in enumerate([(-1, 0), (0, 1), (-1, 0)]):
        val = float(Fraction(w) * f * P)
        nl = y[b] - 0.0
        # G = 0 has no kinetic term: the nonlocal sum alone, one rounding of w (2^-53) and one of the result
        g0 = int(np.argmin([float(k) for k in kin]))
        assert float(kin[g0]) == 0.0
        got = nl[g0]
        assert abs(got.real - vr * val) <= 3 * 2.0 ** -53 * val and abs(got.imag - vi * val) <= 3 * 2.0 ** -53 * val


def test_zero_and_non_finite_bands(lib):
    m = _miller()
    rng = np.random.default_rng(0)
    P = 20
    beta = (rng.standard_normal((P, len(m))) + 1j * rng.standard_normal((P, len(m)))) / np.sqrt(len(m))
    psi = workloads.random_block(len(m), 6, 3)
    psi[1] = 0.0
    psi[3, 11] = np.nan
    psi[4, 700] = -np.inf
    y = _apply(beta, np.eye(P), psi)
    assert np.all(y[1] == 0.0)
    assert np.all(np.isnan(y[3])) and np.all(np.isnan(y[4]))
    assert np.all(np.isfinite(y[[0, 2, 5]]))
    alone = _apply(beta, np.eye(P), psi[[0, 2, 5]])
    assert np.array_equal(y[[0, 2, 5]], alone)
