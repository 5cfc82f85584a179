"""The work that a program built on this library has it do, as cases that can be timed.

A case is one call of a public entry point on a synthetic cell of the kind the benchmark and the tests
use: Gaussian wells for V(r), four s+p projectors per atom, starting orbitals damped by 1/(1+|k+G|^2).

    apply    hpsi_apply on a block of bands (what an eigensolver or a propagator calls)
    gamma    hpsi_apply_gamma, the real-orbital form at k = 0
    kbatch   hpsi_apply_batch over the k-points of one cell
    cells    hpsi_apply_batch over independent cells of different sizes
    eigh     the lowest pairs of a dense reduced problem (complex Hermitian or real symmetric)
    solve    a whole davidson_solve / davidson_solve_gamma from a starting block

In a mixed-precision context H|psi> and the eigenpairs are computed to float32 accuracy and come back
in float64 storage; the program of a mixed case keeps them in float32 and complex64, the types that
carry them (the library's own mixed-precision solver holds its basis the same way).  Eigenvectors are determined up to a phase; the
program fixes it by making the overlap with a given reference vector real and positive.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads
from paper_0906_2569_gb300 import binding as B

TWO_PI = 2.0 * math.pi


def _case(kind, **kw):
    base = {
        "apply": dict(lattice="cubic", a=10.0, ecut=10.0, atoms=2, n1=0, n2=0, n3=0, k=0.0, dense_d=False,
                      bands=16, mixed=False),
        "gamma": dict(lattice="cubic", a=10.0, ecut=10.0, atoms=2, n1=0, n2=0, n3=0, bands=16, mixed=False),
        "kbatch": dict(lattice="fcc", a=10.2, ecut=25.0, atoms=2, points=16, bands=24, shape=3000, mixed=False),
        "cells": dict(cells=32, a_min=8.0, a_max=14.0, ecut=15.0, bands_min=8, bands_max=32, shape=4000, mixed=False),
        "eigh": dict(n=480, wanted=160, real=False),
        "solve": dict(lattice="cubic", a=10.0, ecut=10.0, atoms=2, bands=16, mixed=False, real=False, tol=1e-8),
    }[kind]
    assert set(kw) <= set(base) | {"name"}
    return {"kind": kind, **base, **kw}


def listed():
    return [
        # A small molecule-sized cell with its 16 occupied and few empty bands: the shortest call an
        # eigensolver makes over and over, where launches and latency count.
        _case("apply", name="apply_small_fp64", bands=16),
        # The same cell with a wide block of bands in mixed precision (spectra, many empty states).
        _case("apply", name="apply_wide_mixed", bands=160, mixed=True),
        # A bulk-like cell of 64 atoms, all its occupied bands: the ordinary production block, both precisions,
        # in a box somewhat above the smallest one.
        _case("apply", name="apply_bulk_fp64", a=20.5, ecut=20.0, atoms=64, n1=90, n2=90, n3=90, bands=160),
        _case("apply", name="apply_bulk_mixed", a=20.5, ecut=20.0, atoms=64, n1=90, n2=90, n3=90, bands=160,
              mixed=True),
        # A non-cubic box of an oblique cell off the zone centre, with a D that couples all projectors
        # and an odd number of bands.
        _case("apply", name="apply_oblique_fp64", lattice="fcc", a=10.2, ecut=25.0, atoms=3, n1=27, n2=30, n3=32,
              k=0.2, dense_d=True, bands=37),
        # A large Gamma-only cell (216 atoms): the block that the real-orbital eigensolver applies H to.
        _case("gamma", name="gamma_large_mixed", a=30.0, ecut=25.0, atoms=216, n1=144, n2=144, n3=144, bands=512,
              mixed=True),
        # Real orbitals in float64 on the bulk-like cell in its smallest box, a block of corrections of odd size.
        _case("gamma", name="gamma_bulk_fp64", a=20.5, ecut=20.0, atoms=64, bands=75),
        # Brillouin-zone sampling: 16 k-points with uneven plane-wave counts, mixed precision.
        _case("kbatch", name="kpoints_mixed", mixed=True),
        # A screening run: 32 unrelated small cells with 8 to 32 bands each, float64.
        _case("cells", name="cells_fp64"),
        # The reduced problem of a Rayleigh-Ritz step: four blocks of 160 vectors, the lowest 160 pairs.
        _case("eigh", name="eigh_reduced", n=640, wanted=160),
        # Whole eigensolver calls: the small cell in float64, and real orbitals in mixed precision.
        _case("solve", name="solve_small_fp64"),
        _case("solve", name="solve_real_mixed", bands=32, mixed=True, real=True, tol=1e-5, a=14.0, ecut=12.0, atoms=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds of the listed ones with other cells, cutoffs, block sizes and options."""
    kind = rng.choice(["apply", "apply", "apply", "apply", "gamma", "gamma", "kbatch", "cells", "eigh", "solve"])
    mixed = rng.random() < 0.5
    if kind in ("apply", "gamma"):
        ecut = round(rng.uniform(8.0, 25.0), 2)
        # plane waves from about a thousand to about 40 thousand (160 thousand in the real form)
        npw = math.exp(rng.uniform(math.log(1200.0), math.log(40000.0 if kind == "apply" else 120000.0)))
        a = round((6.0 * math.pi ** 2 * npw) ** (1.0 / 3.0) / math.sqrt(2.0 * ecut), 3)
        atoms = max(1, min(216, int(a ** 3 / 135.0 * rng.uniform(0.5, 1.2))))
        bands = _log(rng, 1, 200)
        while npw * bands * (1 if mixed else 4) > 4.0e6 * (4 if kind == "gamma" else 1):
            bands = max(1, bands // 2)
        if kind == "gamma":
            return _case("gamma", a=a, ecut=ecut, atoms=atoms, bands=bands, mixed=mixed)
        if rng.random() < 0.25 and npw < 6000:
            # off the zone centre, cubic or face-centred (the same volume), a box with three edges of its own
            lattice = rng.choice(["cubic", "fcc"])
            edge = a if lattice == "cubic" else a * 4.0 ** (1.0 / 3.0) / math.sqrt(2.0)
            if lattice == "fcc":
                a = round(a * 4.0 ** (1.0 / 3.0), 3)
            need = 2 * int(edge * math.sqrt(2.0 * ecut) / TWO_PI + 0.5) + 5
            n = [workloads.smooth_235_at_least(need + rng.randrange(0, need)) for _ in range(3)]
            return _case("apply", lattice=lattice, a=a, ecut=ecut, atoms=atoms, n1=n[0], n2=n[1], n3=n[2],
                         k=round(rng.uniform(0.0, 0.3), 3), dense_d=rng.random() < 0.5, bands=min(bands, 64),
                         mixed=mixed)
        return _case("apply", a=a, ecut=ecut, atoms=atoms, bands=bands, mixed=mixed)
    if kind == "kbatch":
        return _case("kbatch", a=round(rng.uniform(7.0, 12.0), 2), ecut=round(rng.uniform(12.0, 25.0), 2),
                     atoms=rng.randint(1, 3), points=rng.randint(2, 20), bands=_log(rng, 4, 40),
                     shape=rng.randrange(1 << 20), mixed=mixed)
    if kind == "cells":
        lo = rng.uniform(7.0, 11.0)
        return _case("cells", cells=rng.randint(3, 32), a_min=round(lo, 2), a_max=round(lo + rng.uniform(0.5, 4.0), 2),
                     ecut=round(rng.uniform(8.0, 15.0), 2), bands_min=4, bands_max=rng.randint(8, 32),
                     shape=rng.randrange(1 << 20), mixed=mixed)
    if kind == "eigh":
        n = _log(rng, 24, 1000)
        return _case("eigh", n=n, wanted=max(1, int(n * rng.uniform(0.2, 0.6))), real=rng.random() < 0.5)
    # block solves of small cells (the solver keeps a basis of up to four blocks)
    ecut = round(rng.uniform(8.0, 12.0), 2)
    a = round(rng.uniform(9.0, 12.0), 3)
    return _case("solve", a=a, ecut=ecut, atoms=rng.randint(2, 5), bands=_log(rng, 4, 40), mixed=mixed,
                 real=rng.random() < 0.5, tol=1e-5 if mixed else 1e-8)


# ---------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _lattice(kind, a):
    if kind == "cubic":
        return np.diag([a, a, a]).astype(np.float64)
    return 0.5 * a * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])


def _atoms(lat, count, rng):
    """Atoms on a jittered grid where one fits the count, else at random positions."""
    edge = round(count ** (1.0 / 3.0))
    if edge ** 3 == count and edge > 1:
        grid = np.stack(np.meshgrid(*[np.arange(edge)] * 3, indexing="ij"), axis=-1).reshape(-1, 3) / edge
        return grid @ lat + rng.uniform(-0.3, 0.3, size=(count, 3))
    return rng.random((count, 3)) @ lat


def _box(case, lat, kpts):
    if case.get("n1"):
        return (case["n1"], case["n2"], case["n3"])
    if case["lattice"] == "cubic":
        n = workloads.cubic_box(case["a"], case["ecut"])
        return (n, n, n)
    # twice the largest Miller index of the sphere on each side of zero, so that no product aliases
    mmax = max(int(np.abs(B.hpsi_gsphere(lat, case["ecut"], k)).max()) for k in kpts)
    n = workloads.smooth_235_at_least(4 * mmax + 1)
    return (n, n, n)


def _potential(lat, atoms, fft):
    """The periodic sum of Gaussian wells -2 exp(-|r - R|^2 / 2) from its Fourier series, on the box."""
    dev = _dev()
    rec = torch.from_numpy(workloads.reciprocal(lat)).to(dev)
    m = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=dev) for n in fft]
    frac = torch.from_numpy(np.asarray(atoms) @ np.linalg.inv(lat)).to(dev)
    ph = [torch.exp(-1j * TWO_PI * m[i][:, None] * frac[None, :, i]) for i in range(3)]
    s = torch.einsum("am,bm,cm->abc", ph[0], ph[1], ph[2]) if len(atoms) < 8 else (
        (ph[0][:, None, :] * ph[1][None, :, :]).reshape(fft[0] * fft[1], -1) @ ph[2].T).reshape(fft)
    g = (m[0][:, None, None, None] * rec[0] + m[1][None, :, None, None] * rec[1] + m[2][None, None, :, None] * rec[2])
    vg = workloads.V_DEPTH * TWO_PI ** 1.5 / abs(np.linalg.det(lat)) * torch.exp(-0.5 * (g * g).sum(-1)) * s
    return torch.fft.ifftn(vg).real.contiguous() * (fft[0] * fft[1] * fft[2])


def _q(lat, k, miller):
    rec = torch.from_numpy(workloads.reciprocal(lat)).to(_dev())
    return torch.from_numpy(np.asarray(k, dtype=np.float64)).to(_dev()) + torch.from_numpy(miller).to(_dev()).double() @ rec


def _projectors(lat, atoms, k, miller):
    q = _q(lat, k, miller)
    radial = torch.exp(-workloads.BETA_ALPHA * (q * q).sum(1))
    phase = torch.exp(-1j * (torch.from_numpy(np.asarray(atoms)).to(_dev()) @ q.T))          # [atom][npw]
    form = torch.stack([radial, q[:, 0] * radial, q[:, 1] * radial, q[:, 2] * radial])    # [4][npw]
    form = form / torch.linalg.vector_norm(form, dim=1, keepdim=True)
    return (phase[:, None, :] * form[None, :, :]).reshape(4 * len(atoms), -1)


def _dmat(count, dense, rng):
    d = workloads.dmat(count)
    if dense:
        b = 0.1 * (rng.standard_normal(d.shape) + 1j * rng.standard_normal(d.shape))
        d = d + (b + b.conj().T) / 2.0
    return d


def _psi(lat, k, miller, bands, gen):
    q = _q(lat, k, miller)
    z = torch.randn(bands, len(miller), dtype=torch.complex128, device=_dev(), generator=gen)
    return (z / (1.0 + (q * q).sum(1))).contiguous()


def _half(psi, npw):
    """The half-sphere coefficients of real orbitals, G = 0 first (real)."""
    h = psi[:, npw // 2:].clone()
    h[:, 0] = h[:, 0].real.to(h.dtype)
    return h


def _cell(case, seed):
    """Everything of one cell (or of one cell's k-points) as the setup call takes it."""
    rng = np.random.default_rng([int(seed), 17])
    lat = _lattice(case["lattice"], case["a"])
    atoms = _atoms(lat, case["atoms"], rng)
    rec = workloads.reciprocal(lat)
    if case["kind"] == "kbatch":
        krng = np.random.default_rng(case["shape"])
        kpts = np.array([workloads.fold_to_bz((krng.random(3) - 0.5) @ rec, rec) for _ in range(case["points"])])
    else:
        kpts = (np.array([[1.0, 0.6, -0.3]]) * case.get("k", 0.0)) @ rec
    fft = _box(case, lat, kpts)
    millers = [B.hpsi_gsphere(lat, case["ecut"], k) for k in kpts]
    return dict(lat=lat, ecut=case["ecut"], kpts=kpts, fft=fft, millers=millers, v=_potential(lat, atoms, fft),
                betas=[_projectors(lat, atoms, k, m) for k, m in zip(kpts, millers)],
                d=_dmat(case["atoms"], case.get("dense_d", False), rng))


def _cell_cases(case):
    """The cells of a screening run: sizes from the case alone."""
    rng = np.random.default_rng(case["shape"])
    return [dict(kind="apply", lattice="cubic", a=float(rng.uniform(case["a_min"], case["a_max"])), ecut=case["ecut"],
                 atoms=int(rng.integers(1, 5)), bands=int(rng.integers(case["bands_min"], case["bands_max"] + 1)))
            for _ in range(case["cells"])]


def _systems(case, seed):
    """The cells of a case with, per problem of the context, its starting block."""
    gen = _gen(2 * int(seed) + 1)
    if case["kind"] == "cells":
        subs = _cell_cases(case)
        cells = [_cell(s, int(seed) * 64 + i) for i, s in enumerate(subs)]
        return cells, [_psi(c["lat"], c["kpts"][0], c["millers"][0], s["bands"], gen) for s, c in zip(subs, cells)]
    c = _cell(case, seed)
    psi = [_psi(c["lat"], k, m, case["bands"], gen) for k, m in zip(c["kpts"], c["millers"])]
    if case["kind"] == "gamma" or case.get("real"):
        psi = [_half(x, len(m)) for x, m in zip(psi, c["millers"])]
    return [c], psi


def _setup(case, cells):
    precision = B.HPSI_MIXED if case["mixed"] else B.HPSI_FP64
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "cells":
        return B.hpsi_setup_cells([c["lat"] for c in cells], [c["ecut"] for c in cells], [c["fft"] for c in cells],
                                  [c["v"].cpu().numpy() for c in cells], [c["betas"][0].cpu().numpy() for c in cells],
                                  [c["d"] for c in cells], precision, stream)
    c = cells[0]
    return B.hpsi_setup(c["lat"], c["ecut"], c["kpts"], c["fft"], c["v"].cpu().numpy(),
                        [b.cpu().numpy() for b in c["betas"]], c["d"], precision, stream)


def _matrix(case, seed):
    """A reduced matrix as a Rayleigh-Ritz step meets it: Ritz values and, above them, the energies of
    the corrections on the diagonal, coupled by a dense Hermitian remainder."""
    n, gen = case["n"], _gen(seed)
    dtype = torch.float64 if case["real"] else torch.complex128
    low = torch.sort(torch.rand(case["wanted"], dtype=torch.float64, device=_dev(), generator=gen))[0] * 3.0 - 2.0
    high = torch.sort(torch.rand(n - case["wanted"], dtype=torch.float64, device=_dev(), generator=gen))[0] * 9.0 + 1.0
    b = torch.randn(n, n, dtype=dtype, device=_dev(), generator=gen) * (0.5 / math.sqrt(n))
    a = b + b.mH
    a += torch.diag(torch.cat([low, high])).to(dtype)
    ref = torch.randn(n, dtype=dtype, device=_dev(), generator=gen)
    return a, ref


def prepare(case, seed):
    if case["kind"] == "eigh":
        a, ref = _matrix(case, seed)
        # any context serves: the reduced problem does not depend on its operator
        ctx = B.hpsi_setup(_lattice("cubic", 6.0), 1.0, np.zeros((1, 3)), (8, 8, 8), np.zeros((8, 8, 8)), None, None,
                           B.HPSI_FP64, torch.cuda.current_stream().cuda_stream)
        # the entry point reads columns: row i of the tensor it is given is column i
        return dict(case=case, ctx=ctx, a=a.T.contiguous(), ref=ref,
                    w=torch.empty(case["wanted"], dtype=torch.float64, device=_dev()),
                    v=torch.empty(case["wanted"], case["n"], dtype=a.dtype, device=_dev()))
    cells, psi = _systems(case, seed)
    state = dict(case=case, ctx=_setup(case, cells), psi=psi, out=[torch.empty_like(x) for x in psi])
    if case["kind"] == "solve":
        state["ref"] = torch.randn(psi[0].shape[1], dtype=torch.complex128, device=_dev(), generator=_gen(seed))
    return state


def _phased(vectors, ref, real):
    """Rows of `vectors` with their free phase (sign, for real ones) fixed against `ref`."""
    dot = vectors @ ref.conj()
    if real:
        return vectors * torch.sgn(dot.real)[:, None]
    return vectors * (dot.conj() / dot.abs())[:, None]


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "eigh":
        call = B.hpsi_eigh_lowest_sym if case["real"] else B.hpsi_eigh_lowest
        call(ctx, state["a"], case["n"], case["n"], case["wanted"], state["w"], state["v"])
        return {"eig": state["w"], "vec": _phased(state["v"], state["ref"], case["real"])}
    if kind == "solve":
        block = state["psi"][0].clone()
        call = B.davidson_solve_gamma if case["real"] else B.davidson_solve
        eig, _, _, _ = call(ctx, 0, block, case["tol"], 200)
        block = _phased(block, state["ref"], case["real"])
        return {"eig": eig.astype(np.float32), "psi": block.to(torch.complex64)} if case["mixed"] else {
            "eig": eig, "psi": block}
    if kind == "apply":
        B.hpsi_apply(ctx, 0, state["psi"][0], state["out"][0])
    elif kind == "gamma":
        B.hpsi_apply_gamma(ctx, 0, state["psi"][0], state["out"][0])
    else:
        B.hpsi_apply_batch(ctx, list(range(len(state["psi"]))), state["psi"], state["out"])
    return [x.to(torch.complex64) for x in state["out"]] if case["mixed"] else state["out"]


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without, and what it should give
# ---------------------------------------------------------------------------------------------------

def _work_apply(npw, nst, npl, fft, nproj, bands, real):
    """Bytes and flops of H on a block: psi read and H psi written once, V, the kinetic diagonal and the projectors once;
    the sphere-pruned line transforms (5 n log2 n each) and two contractions with the projectors."""
    line = [5.0 * n * math.log2(n) for n in fft]
    local = 2.0 * (nst * line[2] + fft[2] * (npl * line[1] + fft[1] * line[0] + fft[0] * fft[1]))
    half = 0.5 if real else 1.0
    nl = 16.0 * nproj * npw * (0.25 if real else 1.0)
    size = 16.0 * (npw * nproj * half + npw * half * bands * 2) + 8.0 * (npw + fft[0] * fft[1] * fft[2])
    return {"bytes": size, "flops": bands * (half * local + nl + 4.0 * npw * half)}


def work(case):
    if case["kind"] == "eigh":
        n, w = case["n"], case["wanted"]
        scale = 1.0 if case["real"] else 4.0
        # reduction to tridiagonal form, back-transformation of the wanted vectors
        return {"bytes": 8.0 * (1 if case["real"] else 2) * (n * n / 2 + n * w),
                "flops": scale * (4.0 * n ** 3 / 3.0 + 2.0 * n * n * w)}
    total = {"bytes": 0.0, "flops": 0.0}
    subs = _cell_cases(case) if case["kind"] == "cells" else [case]
    for s in subs:
        lat = _lattice(s["lattice"], s["a"])
        rec = workloads.reciprocal(lat)
        if case["kind"] == "kbatch":
            krng = np.random.default_rng(case["shape"])
            kpts = np.array([workloads.fold_to_bz((krng.random(3) - 0.5) @ rec, rec) for _ in range(case["points"])])
        else:
            kpts = (np.array([[1.0, 0.6, -0.3]]) * s.get("k", 0.0)) @ rec
        fft = _box(s, lat, kpts)
        for k in kpts:
            m = B.hpsi_gsphere(lat, s["ecut"], k)
            nst, npl = len(np.unique(m[:, :2], axis=0)), len(np.unique(m[:, 0]))
            real = case["kind"] == "gamma" or case.get("real", False)
            w = _work_apply(len(m), nst, npl, fft, 4 * s["atoms"], s["bands"], real)
            if case["kind"] == "solve":
                # a block solve applies H about ten times and works on a basis of about three blocks
                nb = s["bands"]
                w = {"bytes": w["bytes"], "flops": 10.0 * (w["flops"] + 8.0 * 6.0 * nb * nb * len(m) * (0.25 if real else 1.0))}
            total = {key: total[key] + w[key] for key in total}
    return total


def _h_full(cell, ik, psi):
    """H psi on the full sphere with torch in 64 bits: full-box FFTs and dense contractions."""
    fft, m = cell["fft"], torch.from_numpy(cell["millers"][ik]).to(_dev()).long()
    n = fft[0] * fft[1] * fft[2]
    idx = ((m[:, 0] % fft[0]) * fft[1] + m[:, 1] % fft[1]) * fft[2] + m[:, 2] % fft[2]
    q = _q(cell["lat"], cell["kpts"][ik], cell["millers"][ik])
    out = 0.5 * (q * q).sum(1) * psi
    step = max(1, int(2.0e8) // n)
    for b in range(0, len(psi), step):
        x = torch.zeros(len(psi[b:b + step]), n, dtype=torch.complex128, device=_dev())
        x[:, idx] = psi[b:b + step]
        r = torch.fft.ifftn(x.view(-1, *fft), dim=(1, 2, 3), norm="forward") * cell["v"]
        out[b:b + step] += torch.fft.fftn(r, dim=(1, 2, 3), norm="forward").view(-1, n)[:, idx]
        del x, r
    beta = cell["betas"][ik]
    if beta.shape[0]:
        w = (psi @ beta.mH) @ torch.from_numpy(cell["d"]).to(_dev()).T
        out += w @ beta
    return out


def _full(half):
    """Full-sphere coefficients of real orbitals from the half sphere."""
    return torch.cat([half[:, 1:].flip(1).conj(), half], dim=1)


def exact(case, seed):
    if case["kind"] == "eigh":
        a, ref = _matrix(case, seed)
        w, v = torch.linalg.eigh(a.cpu())
        v = v[:, :case["wanted"]].T.contiguous().to(_dev())
        return {"eig": w[:case["wanted"]].to(_dev()), "vec": _phased(v, ref, case["real"])}
    cells, psi = _systems(case, seed)
    if case["kind"] == "solve":
        c = cells[0]
        npw = len(c["millers"][0])
        if npw > 6000:
            return None
        h = torch.cat([_h_full(c, 0, e) for e in torch.eye(npw, dtype=torch.complex128, device=_dev()).split(256)])
        if case["real"]:
            # the orthonormal real basis: G = 0, then (e_G + e_-G)/sqrt2 and (e_G - e_-G)/(i sqrt2)
            nh = (npw + 1) // 2
            u = torch.zeros(npw, npw, dtype=torch.complex128, device=_dev())
            i = torch.arange(1, nh, device=_dev())
            u[0, nh - 1] = 1.0
            u[i, nh - 1 + i] = u[i, nh - 1 - i] = 1.0 / math.sqrt(2.0)
            u[nh - 1 + i, nh - 1 + i] = 1j / math.sqrt(2.0)
            u[nh - 1 + i, nh - 1 - i] = -1j / math.sqrt(2.0)
            # rows of h are H e_G, so the matrix of H is its transpose
            hr = (u.conj() @ h.T @ u.T).real
            w, v = torch.linalg.eigh((hr + hr.T) / 2.0)
            full = v[:, :case["bands"]].T.to(torch.complex128) @ u
            vec = full[:, nh - 1:].contiguous()
        else:
            w, v = torch.linalg.eigh((h.T + h.conj()) / 2.0)
            vec = v[:, :case["bands"]].T.contiguous()
        ref = torch.randn(psi[0].shape[1], dtype=torch.complex128, device=_dev(), generator=_gen(seed))
        return {"eig": w[:case["bands"]].cpu().numpy(), "psi": _phased(vec, ref, case["real"])}
    if case["kind"] == "cells":
        return [_h_full(c, 0, x) for c, x in zip(cells, psi)]
    if case["kind"] == "gamma":
        npw = len(cells[0]["millers"][0])
        return [_h_full(cells[0], 0, _full(psi[0]))[:, npw // 2:].contiguous()]
    return [_h_full(cells[0], i, x) for i, x in enumerate(psi)]
