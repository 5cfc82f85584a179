"""The float64 subspace products of davidson_solve (csrc/subspace_fp64.cu) through whole solves of the 1503-plane-wave cell:
one band, odd block sizes, and blocks large enough for the digit products on the tensor cores; eigenvalues against the dense
oracle's, orthonormal eigenvectors with small residuals of the oracle's H.

Tolerances: the solver stops at residual 1e-8, so an eigenvalue is within 1e-16 / gap of the exact one and the float64
reduced problems round at ~1e-14 Ha: 1e-10 Ha as everywhere; Cholesky QR leaves orthonormality at a few 2^-53
times the block's condition (below 1e3): 1e-12."""
import json
import os

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "eigenvalues.json")


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("nbnd", [1, 5, 33, 130])
def test_solve_block_sizes(lib, nbnd, real):
    import torch
    from paper_0906_2569_gb300 import binding as B
    p = workloads.config3(nbnd)
    k = p.kpts[0]
    m = B.hpsi_gsphere(p.lattice, p.ecut, k)
    npw = len(m)
    vr = workloads.vloc_r(p.lattice, p.atoms, p.fft)
    beta = workloads.beta(p.lattice, p.atoms, k, m)
    d = workloads.dmat(len(p.atoms))
    ctx = B.hpsi_setup(p.lattice, p.ecut, [k], p.fft, vr, [beta], d, B.HPSI_FP64,
                       torch.cuda.current_stream().cuda_stream)
    psi = workloads.psi0(p.lattice, k, m, nbnd, p.psi_seed)
    if real:
        psi = psi[:, npw // 2:].copy()
        psi[:, 0] = psi[:, 0].real
    x = torch.from_numpy(psi).cuda()
    eig, _, res, _ = (B.davidson_solve_gamma if real else B.davidson_solve)(ctx, 0, x, 1e-8, 200)
    ctx.close()
    ref = np.asarray(json.load(open(GOLDEN))["c3"]["eigenvalues"])[:nbnd]
    assert np.max(np.abs(eig - ref)) < 1e-10
    v = x.cpu().numpy()
    if real:
        v = np.concatenate([v[:, 1:][:, ::-1].conj(), v], axis=1)
    assert np.max(np.abs(v.conj() @ v.T - np.eye(nbnd))) < 1e-12
    hv = oracle.hamiltonian.hpsi(p.lattice, k, m, p.fft, vr, beta, d, v)
    assert np.max(np.linalg.norm(hv - eig[:, None] * v, axis=1)) < 1e-8 + 1e-12


@pytest.mark.parametrize("nbnd,real", [(2, True), (33, True), (240, True), (2, False), (33, False), (130, False)])
def test_mixed_vectors_refined(lib, nbnd, real):
    """The float32 basis's vectors leave the solver refined in float64: rows of a float32 block are orthogonal to ~3e-7, refined ones
    to second order in the mixing taken out (1e-5 noise over gap), summed over the block: 1e-10 a band."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    p = workloads.config3(nbnd)
    k = p.kpts[0]
    m = B.hpsi_gsphere(p.lattice, p.ecut, k)
    npw = len(m)
    vr = workloads.vloc_r(p.lattice, p.atoms, p.fft)
    ctx = B.hpsi_setup(p.lattice, p.ecut, [k], p.fft, vr, [workloads.beta(p.lattice, p.atoms, k, m)],
                       workloads.dmat(len(p.atoms)), B.HPSI_MIXED, torch.cuda.current_stream().cuda_stream)
    psi = workloads.psi0(p.lattice, k, m, nbnd, p.psi_seed)
    if real:
        psi = psi[:, npw // 2:].copy()
        psi[:, 0] = psi[:, 0].real
    x = torch.from_numpy(psi).cuda()
    eig, _, res, _ = (B.davidson_solve_gamma if real else B.davidson_solve)(ctx, 0, x, 1e-5, 200)
    ctx.close()
    ref = np.asarray(json.load(open(GOLDEN))["c3"]["eigenvalues"])[:nbnd]
    assert np.max(np.abs(eig - ref)) < 1e-6
    assert np.max(res) < 1e-5
    v = x.cpu().numpy()
    if real:
        v = np.concatenate([v[:, 1:][:, ::-1].conj(), v], axis=1)
    o = v.conj() @ v.T
    assert np.max(np.abs(o - np.diag(np.diag(o)))) < 1e-10 * max(nbnd, 10)
