"""The fixed-point local term of float64 contexts (csrc/local_fixed.cu) against the oracle: every pair of radices, boxes
with three different edges, plane counts and chunk remainders at the edges of the tiles, inputs over the
float64 exponent range, zeros and non-finite values.

Tolerance: H|psi> is summed in float64, so its rounding alone is 2^-53 of |H psi|; the transforms of either
side add a few 2^-53 of |V psi| (at most ~sqrt(log2 N) roundings each): 2e-15 of the norm of H psi covers both."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = 2e-15


def _case(lib, fft, a, ecut, k=(0.0, 0.0, 0.0), lattice=None, scale=1.0, nb=3, v=None, psi=None):
    import torch
    from paper_0906_2569_gb300 import binding as B
    lat = np.diag([a, a, a]).astype(float) if lattice is None else np.asarray(lattice, dtype=float)
    k = np.asarray(k, dtype=float)
    m = B.hpsi_gsphere(lat, ecut, k)
    rng = np.random.default_rng(fft[0] * 1000 + fft[2])
    vr = rng.standard_normal(fft) if v is None else v
    x = scale * workloads.random_block(len(m), nb, 5) if psi is None else psi
    ctx = B.hpsi_setup(lat, ecut, [k], fft, vr, None, None, B.HPSI_FP64, torch.cuda.current_stream().cuda_stream)
    xd = torch.from_numpy(x).cuda()
    y = torch.full_like(xd, float("nan"))
    B.hpsi_apply(ctx, 0, xd, y)
    B.hpsi_sync(ctx)
    n = B.hpsi_kernel_stats(ctx, B.KERNELS.index("xvx_y"))[0]
    ctx.close()
    assert n >= 1
    return lat, k, m, vr, x, y.cpu().numpy()


def _check(lib, fft, a, ecut, **kw):
    lat, k, m, vr, x, y = _case(lib, fft, a, ecut, **kw)
    none = np.zeros((0, len(m)), dtype=complex)
    ref = oracle.hamiltonian.hpsi(lat, k, m, fft, vr, none, np.zeros((0, 0), dtype=complex), x)
    for b in range(len(x)):
        top = np.max(np.abs(ref[b]))   # norms of 1e290 or 1e-290 would leave the float64 range
        err = np.linalg.norm((y[b] - ref[b]) / top) / np.linalg.norm(ref[b] / top)
        assert err < TOL, f"box {fft} band {b}: {err:.2e}"


# every edge with a two-factor split, smallest first (a sphere that fills about half the edge)
@pytest.mark.parametrize("n", [8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80,
                               81, 90, 96, 100, 108, 120, 128, 135, 144, 150, 160])
def test_cubic_edges(lib, n):
    mmax = max(1, (n - 1) // 4)
    a = 2.0 * np.pi * (mmax + 0.3) / np.sqrt(2.0 * 8.0)
    _check(lib, (n, n, n), a, 8.0, nb=3 if n < 100 else 1)


@pytest.mark.parametrize("fft,a,ecut,k", [
    ((8, 25, 12), 4.0, 5.0, (0.1, 0.0, 0.2)), ((27, 30, 32), 7.2, 25.0, (0.2, -0.1, 0.3)),
    ((32, 27, 30), 7.2, 25.0, (0.0, 0.0, 0.0)), ((50, 15, 16), 4.9, 6.0, (0.0, 0.1, 0.0)),
    ((9, 160, 10), 3.7, 5.0, (0.0, 0.0, 0.0)), ((96, 10, 128), 4.0, 5.0, (0.3, 0.0, 0.0)),
    # a tight box: the sphere reaches the box's edge, so all sticks and planes but one are filled
    ((15, 15, 15), 10.0, 9.8, (0.0, 0.0, 0.0)), ((25, 25, 27), 12.0, 19.5, (0.0, 0.0, 0.0))])
def test_unequal_and_tight_boxes(lib, fft, a, ecut, k):
    _check(lib, fft, a, ecut, k=k)
    if len(set(fft)) > 1 and ecut == 25.0:
        lat = 0.5 * 10.2 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])
        _check(lib, fft, a, ecut, k=k, lattice=lat)


def test_generic_only_edge_still_runs(lib):
    """125 = 5 x 25 has no pair of codelets: the generic radix kernels serve it."""
    _check(lib, (125, 125, 125), 2.0 * np.pi * 20.3 / 4.0, 8.0, nb=1)


@pytest.mark.parametrize("scale", [1e-290, 1e-30, 1e30, 1e290])
def test_exponent_range(lib, scale):
    _check(lib, (36, 36, 36), 10.0, 15.0, scale=scale)


def test_spread_of_magnitudes(lib):
    """One dominant coefficient, and bands that differ by 1e200: the error is relative to each band's own norm."""
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(np.diag([10.0] * 3), 10.0, np.zeros(3))
    x = workloads.random_block(len(m), 4, 3)
    x[0] *= 1e-12
    x[0, 700] = 1.0
    x[1] *= 1e-200
    x[2] *= 1e200
    x[3, : len(m) // 2] = 0.0
    _check(lib, (32, 32, 32), 10.0, 10.0, psi=x)


def test_zero_and_non_finite(lib):
    """A zero band gives exact zeros; a NaN or infinity makes its whole band NaN and touches no other band."""
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(np.diag([10.0] * 3), 10.0, np.zeros(3))
    x = workloads.random_block(len(m), 5, 3)
    x[1] = 0.0
    x[2, 5] = np.nan
    x[4, 900] = np.inf
    lat, k, m, vr, x, y = _case(lib, (32, 32, 32), 10.0, 10.0, psi=x)
    assert np.all(y[1] == 0.0)
    assert np.all(np.isnan(y[2])) and np.all(np.isnan(y[4]))
    none = np.zeros((0, len(m)), dtype=complex)
    ref = oracle.hamiltonian.hpsi(lat, k, m, (32, 32, 32), vr, none, np.zeros((0, 0), dtype=complex), x[[0, 3]])
    for b, r in zip((0, 3), ref):
        assert np.linalg.norm(y[b] - r) / np.linalg.norm(r) < TOL


def test_zero_potential_is_exact(lib):
    """V = 0: H psi is the kinetic diagonal (read off a band of ones) times psi, bit for bit."""
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(np.diag([9.3] * 3), 12.0, np.zeros(3))
    x = workloads.random_block(len(m), 3, 5)
    x[0] = 1.0
    y = _case(lib, (30, 30, 30), 9.3, 12.0, v=np.zeros((30, 30, 30)), psi=x)[-1]
    assert np.array_equal(y.real, y[0].real * x.real) and np.array_equal(y.imag, y[0].real * x.imag)
