"""Eigenvalues and eigenvectors of the reduced problem where the multisection and the inverse iteration change form: block
sizes on both sides of one and two wanted values per SM, the smallest orders, and norms far from one.

Tolerances, relative to the matrix norm: the reduction, the Sturm counts and the back-transformation are each a few
rounding errors of float64 accumulated over n steps; 4 n 2^-53 + 1e-14 covers them for eigenvalues and
residuals, and orthonormality is restored by a Newton-Schulz step to the same order."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    import torch
    from paper_0906_2569_gb300 import binding as B
    p = workloads.config1()
    k = p.kpts[0]
    m = B.hpsi_gsphere(p.lattice, p.ecut, k)
    c = B.hpsi_setup(p.lattice, p.ecut, [k], p.fft, workloads.vloc_r(p.lattice, p.atoms, p.fft),
                     [workloads.beta(p.lattice, p.atoms, k, m)], workloads.dmat(len(p.atoms)), B.HPSI_FP64,
                     torch.cuda.current_stream().cuda_stream)
    yield c
    c.close()


@pytest.mark.parametrize("n,nwant,scale", [(1, 1, 1.0), (2, 2, 1.0), (3, 1, 1e-6), (31, 31, 1.0), (65, 16, 1e3), (160, 152, 1.0),
                                           (160, 153, 1.0), (310, 304, 1.0), (310, 305, 1.0), (64, 16, 1e-15),
                                           (64, 64, 1e15)])
def test_lowest_pairs(ctx, n, nwant, scale):
    import torch
    from paper_0906_2569_gb300 import binding as B
    a = workloads.hermitian_matrix(n, 1000 * n + nwant)
    ref = np.linalg.eigvalsh(a)
    norm = np.max(np.abs(ref))
    w = torch.empty(nwant, dtype=torch.float64, device="cuda")
    v = torch.empty((nwant, n), dtype=torch.complex128, device="cuda")
    B.hpsi_eigh_lowest(ctx, torch.from_numpy(np.ascontiguousarray(a.T) * scale).cuda(), n, n, nwant, w, v)
    w, x = w.cpu().numpy() / scale, v.cpu().numpy().T
    tol = 4 * n * 2.0 ** -53 + 1e-14
    assert np.max(np.abs(w - ref[:nwant])) < tol * norm
    assert np.max(np.linalg.norm(a @ x - x * w, axis=0)) < tol * norm
    assert np.max(np.abs(x.conj().T @ x - np.eye(nwant))) < tol
