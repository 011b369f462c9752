"""The measured workloads of the library: what a program asks of it, through the
calls of paper_2009_01967_gb300, from one-atom crystals to 864-atom supercells.

Every case is a dict of plain values with a "kind" (the call or calls made), a
cell, a q-mesh or a list of supercells, and the options of the call.  Cells are
fcc Lennard-Jones crystals (a = 5.26 A, cutoff 8.5 A, the potential of the
repository's configurations):

  ar      the one-atom primitive cell
  l11     the two-atom L1_1 binary
  alloy   n1 x n2 x n3 conventional cells (4 atoms each), masses 28.09 / 72.63
          shuffled by the seed, with a 2 % isotope spread

A program keeps one library context, its system (host arrays, as the library
takes them) and, where a stage starts from earlier results, the frequencies,
eigenvectors and linewidths on the device.  Linewidths asked for in one of the
single-precision modes ("fp32", "bf16split") are kept as float32, FP64 ones as
float64.
"""

from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2009_01967_gb300 as kk

A_FCC, M_AR, M_LIGHT, M_HEAVY = 5.26, 39.95, 28.09, 72.63
LJ_EPS, LJ_SIG, LJ_CUT = 0.0104, 3.4, 8.5
NU_MIN, DEGEN_TOL, N_SIGMA = 0.01, 1e-5, 3.0

# CODATA 2018 values for the 64-bit results of exact()
_E, _AMU, _KB, _HBAR = 1.602176634e-19, 1.66053906660e-27, 1.380649e-23, 1.054571817e-34
EV_A2_AMU = _E / _AMU * 1e-4                 # eV / (A^2 amu) in ps^-2
KB_EV, HBAR_EV_PS = _KB / _E, _HBAR / _E * 1e12


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # kappa of a small crystal whose linewidths are at hand: the smallest call, bound by latency
        {"name": "kappa_rta_l11", "kind": "kappa_rta", "cell": "l11", "mesh": "6x6x6", "T": 300.0, "sigma": 0.1},
        # the whole path for solid argon in FP64: the smallest complete calculation
        {"name": "step_ar_fp64", "kind": "step", "cell": "ar", "mesh": "6x6x6", "T": 50.0, "sigma": 0.1,
         "precision": "fp64", "delta": "gaussian"},
        # linewidths of a two-atom compound on a dense mesh: the largest number of momentum pairs
        {"name": "linewidths_l11_fp32", "kind": "linewidths", "cell": "l11", "mesh": "24x24x24", "T": 300.0,
         "sigma": 0.05, "precision": "fp32", "delta": "gaussian"},
        # reference-precision linewidths of a middle-sized cell on a coarse mesh
        {"name": "linewidths_alloy8_fp64", "kind": "linewidths", "cell": "alloy", "size": "2x1x1", "mesh": "4x4x4",
         "T": 300.0, "sigma": 0.1, "precision": "fp64", "delta": "gaussian"},
        # tensor-core linewidths of a 32-atom cell on a coarse mesh, as in a mesh convergence test
        {"name": "linewidths_alloy32_split", "kind": "linewidths", "cell": "alloy", "size": "2x2x2", "mesh": "4x4x4",
         "T": 300.0, "sigma": 0.05, "precision": "bf16split", "delta": "gaussian"},
        # the whole path of the 32-atom disordered cell on the 8^3 mesh (the benchmark's workload)
        {"name": "step_alloy32_split", "kind": "step", "cell": "alloy", "size": "2x2x2", "mesh": "8x8x8", "T": 300.0,
         "sigma": 0.05, "precision": "bf16split", "delta": "gaussian"},
        # frequencies, eigenvectors and group velocities of the 32-atom cell on the 8^3 mesh
        {"name": "phonons_alloy32", "kind": "phonons", "cell": "alloy", "size": "2x2x2", "mesh": "8x8x8"},
        # Gamma-only linewidths of one 256-atom supercell
        {"name": "linewidths_cell256_split", "kind": "linewidths_cells", "cells": "4", "T": 300.0, "sigma": 0.05,
         "precision": "bf16split", "delta": "gaussian"},
        # the whole path of a batch of disordered supercells of 108, 256 and 500 atoms
        {"name": "step_cells_split", "kind": "step_cells", "cells": "3,3,3,3,4,4,4,4,5,5,5,5", "T": 300.0,
         "sigma": 0.05, "precision": "bf16split", "delta": "gaussian"},
        # quasi-harmonic Green-Kubo conductivity of the 864-atom supercell
        {"name": "qhgk_cell864", "kind": "qhgk", "cells": "6", "T": 300.0},
        # conductivity from the full linearised transport equation of a two-atom compound
        {"name": "bte_l11", "kind": "bte", "cell": "l11", "mesh": "6x6x6", "T": 300.0, "sigma": 0.1},
        # three-phonon phase space of the 32-atom cell, the screening quantity before any linewidth
        {"name": "phase_space_alloy32", "kind": "phase_space", "cell": "alloy", "size": "2x2x2", "mesh": "6x6x6",
         "T": 300.0, "sigma": 0.05, "precision": "fp32", "delta": "gaussian"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_mesh(rng, lo, hi, nq_max=1 << 30):
    while True:
        m = _log_int(rng, lo, hi)
        mesh = [min(hi, max(1, m + rng.choice([-1, 0, 0, 1]))) for _ in range(3)]
        if math.prod(mesh) <= nq_max:
            return "x".join(str(x) for x in mesh)


def draw(rng):
    kind = rng.choice(["kappa_rta", "step", "step_alloy", "linewidths_small", "linewidths_alloy", "linewidths_split",
                       "phonons", "linewidths_cells", "step_cells", "qhgk", "bte", "phase_space"])
    opt = {"T": round(rng.uniform(50.0, 600.0), 1), "sigma": round(rng.uniform(0.04, 0.2), 3)}
    delta = {"delta": rng.choice(["gaussian", "gaussian", "lorentzian", "triangular"])}
    if kind == "kappa_rta":
        if rng.random() < 0.5:
            return {"kind": kind, "cell": rng.choice(["ar", "l11"]), "mesh": _draw_mesh(rng, 3, 24), **opt}
        return {"kind": kind, "cell": "alloy", "size": rng.choice(["2x1x1", "2x2x1", "2x2x2"]),
                "mesh": _draw_mesh(rng, 2, 6), **opt}
    if kind == "step":
        return {"kind": "step", "cell": rng.choice(["ar", "l11"]), "mesh": _draw_mesh(rng, 3, 10),
                "precision": rng.choice(["fp64", "fp32"]), **opt, **delta}
    if kind == "step_alloy":
        return {"kind": "step", "cell": "alloy", "size": "2x2x2", "mesh": _draw_mesh(rng, 2, 7),
                "precision": "bf16split", **opt, **delta}
    if kind == "linewidths_small":
        return {"kind": "linewidths", "cell": rng.choice(["ar", "l11"]), "mesh": _draw_mesh(rng, 3, 20),
                "precision": rng.choice(["fp32", "fp32", "bf16split"]), **opt, **delta}
    if kind == "linewidths_alloy":
        size, top = rng.choice([("2x1x1", 64), ("2x2x1", 36), ("2x2x2", 18)])
        return {"kind": "linewidths", "cell": "alloy", "size": size, "mesh": _draw_mesh(rng, 2, 4, top),
                "precision": rng.choice(["fp64", "fp32"]), **opt, **delta}
    if kind == "linewidths_split":
        return {"kind": "linewidths", "cell": "alloy", "size": rng.choice(["2x3x1", "2x2x2", "7x1x1"]),
                "mesh": _draw_mesh(rng, 1, 6), "precision": "bf16split", **opt, **delta}
    if kind == "phonons":
        return {"kind": kind, "cell": "alloy", "size": rng.choice(["2x1x1", "2x2x1", "2x3x1", "2x2x2"]),
                "mesh": _draw_mesh(rng, 2, 8)}
    if kind == "linewidths_cells":
        cells = [rng.choice(["3", "4x3x3", "4x4x3", "3x3x5", "4"]) for _ in range(rng.randint(1, 2))]
        return {"kind": kind, "cells": ",".join(cells), "precision": "bf16split", **opt, **delta}
    if kind == "step_cells":
        cells = [rng.choice(["3", "3x4x3", "4", "4x4x5"]) for _ in range(rng.randint(1, 5))]
        return {"kind": kind, "cells": ",".join(cells), "precision": "bf16split", **opt, **delta}
    if kind == "qhgk":
        cells = [rng.choice(["3", "4x3x3", "4", "5x4x4", "5"]) for _ in range(rng.randint(1, 3))]
        return {"kind": kind, "cells": ",".join(cells), "T": opt["T"]}
    if kind == "bte":
        return {"kind": kind, "cell": rng.choice(["ar", "l11"]), "mesh": _draw_mesh(rng, 3, 6), "T": opt["T"],
                "sigma": round(rng.uniform(0.1, 0.2), 3)}
    precision, top = rng.choice([("fp32", 6), ("fp64", 4)])
    return {"kind": "phase_space", "cell": "alloy", "size": rng.choice(["2x1x1", "2x2x1", "2x2x2"]),
            "mesh": _draw_mesh(rng, 2, top), "precision": precision, **opt, **delta}


# ---------------------------------------------------------------- systems
def _ints(text, sep="x"):
    return [int(x) for x in str(text).split(sep)]


def _cubic(text):
    n = _ints(text)
    return tuple(n * 3 if len(n) == 1 else n)


@functools.lru_cache(maxsize=32)
def _crystal(cell, size):
    """Lattice, positions and analytic Lennard-Jones force constants (home atom
    first), everything but the masses: made once per cell shape."""
    if cell == "ar":
        lat = 0.5 * A_FCC * np.array([[0.0, 1, 1], [1, 0, 1], [1, 1, 0]])
        pos = np.zeros((1, 3))
    elif cell == "l11":
        lat = 0.5 * A_FCC * np.array([[1.0, -1, 0], [0, 1, -1], [1, 2, 1]])
        pos = 0.5 * A_FCC * np.array([[0.0, 0, 0], [1, 1, 0]])
    else:
        n = size
        basis = 0.5 * A_FCC * np.array([[0.0, 0, 0], [0, 1, 1], [1, 0, 1], [1, 1, 0]])
        g = np.stack(np.meshgrid(*[np.arange(x) for x in n[::-1]], indexing="ij"), -1).reshape(-1, 3)[:, ::-1]
        lat = A_FCC * np.diag(np.array(n, float))
        pos = (A_FCC * g[:, None, :] + basis[None]).reshape(-1, 3)
    vol = abs(np.linalg.det(lat))
    reach = []
    for k in range(3):
        width = vol / np.linalg.norm(np.cross(lat[(k + 1) % 3], lat[(k + 2) % 3]))
        reach.append(int(math.ceil(LJ_CUT / width)) + 1)
    cells = np.stack(np.meshgrid(*[np.arange(-r, r + 1) for r in reach], indexing="ij"), -1).reshape(-1, 3)
    shift = cells @ lat
    ii, jj, nn, rr = [], [], [], []
    for i, x in enumerate(pos):
        d = pos[None] + shift[:, None] - x
        r2 = (d * d).sum(-1)
        c, j = np.nonzero((r2 < LJ_CUT ** 2) & (r2 > 1e-12))
        ii.append(np.full(c.size, i))
        jj.append(j)
        nn.append(cells[c])
        rr.append(d[c, j])
    i, j, n, r = np.concatenate(ii), np.concatenate(jj), np.concatenate(nn), np.concatenate(rr)
    d = np.linalg.norm(r, axis=1)
    e = r / d[:, None]
    s6 = (LJ_SIG / d) ** 6
    v1 = 4 * LJ_EPS * (-12 * s6 * s6 + 6 * s6) / d
    v2 = 4 * LJ_EPS * (156 * s6 * s6 - 42 * s6) / d ** 2
    v3 = 4 * LJ_EPS * (-2184 * s6 * s6 + 336 * s6) / d ** 3
    one = np.eye(3)
    ee = e[:, :, None] * e[:, None, :]
    K = v2[:, None, None] * ee + (v1 / d)[:, None, None] * (one - ee)
    a = (v3 - 3 * v2 / d + 3 * v1 / d ** 2)[:, None, None, None]
    b = (v2 / d - v1 / d ** 2)[:, None, None, None]
    T = a * ee[..., None] * e[:, None, None, :] + b * (one[None, :, :, None] * e[:, None, None, :] +
                                                       one[None, :, None, :] * e[:, None, :, None] +
                                                       one[None, None, :, :] * e[:, :, None, None])
    na = len(pos)
    Ks, Ts = np.zeros((na, 3, 3)), np.zeros((na, 3, 3, 3))
    np.add.at(Ks, i, K)
    np.add.at(Ts, i, T)
    z, ic, jc, h = np.zeros_like(n), i[:, None], j[:, None], np.arange(na)[:, None]
    zh = np.zeros((na, 3), n.dtype)
    fc2_idx = np.concatenate([np.hstack([h, h, zh]), np.hstack([ic, jc, n])])
    fc2 = np.concatenate([Ks, -K])
    fc3_idx = np.concatenate([np.hstack([h, h, zh, h, zh]), np.hstack([ic, ic, z, jc, n]),
                              np.hstack([ic, jc, n, ic, z]), np.hstack([ic, jc, n, jc, n])])
    fc3 = np.concatenate([-Ts, T, T, -T])
    o2, o3 = np.lexsort(fc2_idx.T[::-1]), np.lexsort(fc3_idx.T[::-1])
    return (lat, pos, np.ascontiguousarray(fc2_idx[o2], np.int32), np.ascontiguousarray(fc2[o2]),
            np.ascontiguousarray(fc3_idx[o3], np.int32), np.ascontiguousarray(fc3[o3]))


def _system(cell, size, rng):
    lat, pos, i2, f2, i3, f3 = _crystal(cell, size)
    n = len(pos)
    if cell == "ar":
        m = np.full(1, M_AR) * (1.0 + 0.02 * (rng.random() - 0.5))
    elif cell == "l11":
        m = np.array([M_LIGHT, M_HEAVY]) * (1.0 + 0.02 * (rng.random(2) - 0.5))
    else:
        heavy = rng.uniform(0.1, 0.5) if n > 32 else 0.5
        m = np.where(rng.permutation(n) < max(1, round(heavy * n)), M_HEAVY, M_LIGHT)
        m = m * (1.0 + 0.02 * (rng.random(n) - 0.5))
    return SimpleNamespace(masses=m, positions=pos, lattice=lat, fc2_idx=i2, fc2=f2, fc3_idx=i3, fc3=f3)


def _systems(case, seed):
    rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 17])
    if "cells" in case:
        return [_system("alloy", _cubic(c), rng) for c in case["cells"].split(",")]
    return [_system(case["cell"], _cubic(case.get("size", "1")), rng)]


# ------------------------------------------------- 64-bit phonons, in plain torch
def _fractions(mesh):
    return np.stack(np.meshgrid(*[np.arange(m) for m in mesh], indexing="ij"), -1).reshape(-1, 3)


def _flat(k, mesh):
    k = np.mod(k, mesh)
    return (k[..., 0] * mesh[1] + k[..., 1]) * mesh[2] + k[..., 2]


def _qpoints(s, mesh):
    return (_fractions(mesh) / np.array(mesh, float)) @ (2 * np.pi * np.linalg.inv(s.lattice).T)


def _cuda(x, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")


def _dynmat(s, q, weight=None):
    """sum over blocks of Phi2 / sqrt(m m') [times weight] exp(-i q.R), [nq, nb, nb]."""
    nb, n = 3 * len(s.masses), s.fc2_idx
    blk = s.fc2 / np.sqrt(s.masses[n[:, 0]] * s.masses[n[:, 1]])[:, None, None]
    R = n[:, 2:5] @ s.lattice
    at = ((3 * n[:, 0, None] + np.arange(3))[:, :, None] * nb + (3 * n[:, 1, None] + np.arange(3))[:, None, :])
    blk = blk if weight is None else blk * weight[:, None, None]
    blk, at = torch.as_tensor(blk.reshape(-1, 9)), torch.as_tensor(at.reshape(-1))
    # on the host, where the sums have one order: degenerate eigenvectors follow every bit
    out = torch.zeros((nb * nb, len(q)), dtype=torch.complex128)
    step = max(1, (1 << 24) // max(1, at.numel()))
    for x in range(0, len(q), step):
        arg = torch.as_tensor(R @ q[x:x + step].T)
        ph = torch.polar(torch.ones_like(arg), -arg)
        out[:, x:x + step] = torch.zeros((nb * nb, arg.shape[1]), dtype=torch.complex128).index_add_(
            0, at, (blk[:, :, None] * ph[:, None, :]).reshape(at.numel(), -1))
    out = out.T.contiguous().cuda()
    return out.reshape(len(q), nb, nb)


def _phonons(s, mesh):
    """nu [nq, nb] (THz) and eigvec [nq, nb, nb] (row = mode) with eigvec(-q) = conj eigvec(q)."""
    k = _fractions(mesh)
    nq, nb = len(k), 3 * len(s.masses)
    neg = _flat(-k, mesh)
    rep = np.nonzero(neg >= np.arange(nq))[0]
    D = _dynmat(s, _qpoints(s, mesh)[rep])
    lam = torch.empty((nq, nb), dtype=torch.float64, device="cuda")
    eig = torch.empty((nq, nb, nb), dtype=torch.complex128, device="cuda")
    for sel, real in ((rep[neg[rep] == rep], True), (rep[neg[rep] > rep], False)):
        if not len(sel):
            continue
        M = D[torch.as_tensor(np.searchsorted(rep, sel), device="cuda")]
        M = M.real.contiguous() if real else M
        M = 0.5 * (M + M.transpose(-1, -2).conj())
        w, V = torch.linalg.eigh(M) if nb > 96 else torch.linalg.eigh(M.cpu())
        w, V = w.cuda(), V.cuda().transpose(-1, -2).to(torch.complex128)
        sel_t, neg_t = torch.as_tensor(sel, device="cuda"), torch.as_tensor(neg[sel], device="cuda")
        lam[sel_t] = w
        eig[sel_t] = V
        lam[neg_t] = w
        eig[neg_t] = V if real else V.conj()
    w2 = lam * EV_A2_AMU
    return torch.sign(w2) * w2.abs().sqrt() / (2 * math.pi), eig.contiguous()


# ---------------------------------------------------------------- prepare and run
_CTX = None


def _context():
    global _CTX
    if _CTX is None:
        _CTX = kk.Context(torch.cuda.current_device())
        _CTX.set_stream(torch.cuda.current_stream().cuda_stream)
    return _CTX


def _options(case):
    return kk.Options(temperature_K=case["T"], sigma_thz=case.get("sigma", 0.05), n_sigma=N_SIGMA,
                      omega_min_thz=NU_MIN, degen_tol_thz=DEGEN_TOL, precision=case.get("precision", "fp64"),
                      delta=case.get("delta", "gaussian"))


def _model_gamma(nu, seed):
    """Linewidths as they come out for these crystals: about 0.05 nu^2 ps^-1 with scatter."""
    g = torch.Generator(device="cpu").manual_seed(int(seed) & 0x7FFFFFFF)
    r = torch.rand(nu.shape, generator=g, dtype=torch.float64).to(nu.device)
    return torch.where(nu > NU_MIN, 0.05 * nu * nu * (0.5 + r), torch.zeros_like(nu))


def prepare(case, seed):
    st = SimpleNamespace(case=case, ctx=_context(), systems=_systems(case, seed))
    kind = case["kind"]
    st.mesh = (1, 1, 1) if "cells" in case else tuple(_ints(case["mesh"]))
    st.nq = math.prod(st.mesh)
    st.nbs = [3 * len(s.masses) for s in st.systems]
    st.opt = _options(case) if "T" in case else None
    if kind in ("kappa_rta", "linewidths", "linewidths_cells", "qhgk", "bte", "phase_space"):
        ph = [_phonons(s, st.mesh) for s in st.systems]
        st.nu = torch.cat([p[0].reshape(-1) for p in ph])
        st.eig = torch.cat([p[1].reshape(-1) for p in ph])
        del ph
    if kind in ("kappa_rta", "qhgk"):
        st.gamma = _model_gamma(st.nu, seed)
        if kind == "kappa_rta":
            st.gamma = _average(st.nu.reshape(st.nq, -1), st.gamma.reshape(st.nq, -1)).reshape(-1).contiguous()
    return st


def _kept(gamma, case):
    return gamma if case.get("precision", "fp64") == "fp64" else gamma.to(torch.float32)


def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def run(st):
    kind, ctx, s, nq = st.case["kind"], st.ctx, st.systems, st.nq
    nb = st.nbs[0]
    if kind == "kappa_rta":
        return {"kappa": kk.kald_kappa_rta(ctx, s[0], st.mesh, st.nu, st.eig, st.gamma, st.opt, kappa=_empty(3, 3))}
    if kind == "step":
        nu, eig = _empty(nq, nb), _empty(nq, nb, nb, dtype=torch.complex128)
        kk.kald_phonons(ctx, s[0], st.mesh, nu_thz=nu, eigvec=eig, want_vel=False)
        g, _ = kk.kald_linewidths(ctx, s[0], st.mesh, nu, eig, st.opt, gamma=_empty(nq * nb))
        kappa = kk.kald_kappa_rta(ctx, s[0], st.mesh, nu, eig, g, st.opt, kappa=_empty(3, 3))
        return {"nu2": nu * nu.abs(), "gamma": _kept(g, st.case), "kappa": _kept(kappa, st.case)}
    if kind == "linewidths":
        g, count = kk.kald_linewidths(ctx, s[0], st.mesh, st.nu, st.eig, st.opt, gamma=_empty(nq * nb))
        return {"gamma": _kept(g, st.case), "triplets": list(count)}
    if kind == "phonons":
        nu, eig, vel = _empty(nq, nb), _empty(nq, nb, nb, dtype=torch.complex128), _empty(nq, nb, 3)
        kk.kald_phonons(ctx, s[0], st.mesh, nu_thz=nu, eigvec=eig, vel=vel)
        return _phonon_outputs(nu, eig, vel)
    if kind == "linewidths_cells":
        g, count = kk.kald_linewidths(ctx, s, st.mesh, st.nu, st.eig, st.opt, gamma=_empty(sum(st.nbs)))
        return {"gamma": _kept(g, st.case), "triplets": list(count)}
    if kind == "step_cells":
        nu, eig = _empty(sum(st.nbs)), _empty(sum(n * n for n in st.nbs), dtype=torch.complex128)
        kk.kald_phonons_batch(ctx, s, nu_thz=nu, eigvec=eig)
        g, _ = kk.kald_linewidths(ctx, s, st.mesh, nu, eig, st.opt, gamma=_empty(sum(st.nbs)))
        kappa, _ = kk.kald_kappa_qhgk(ctx, s, nu, eig, g, st.opt, kappa=_empty(len(s), 3, 3))
        return {"nu2": nu * nu.abs(), "gamma": _kept(g, st.case), "kappa": _kept(kappa, st.case)}
    if kind == "qhgk":
        kappa, _ = kk.kald_kappa_qhgk(ctx, s, st.nu, st.eig, st.gamma, st.opt, kappa=_empty(len(s), 3, 3))
        return {"kappa": kappa}
    if kind == "bte":
        kappa, _ = kk.kald_kappa_bte(ctx, s[0], st.mesh, st.nu, st.eig, st.opt, tol=1e-11, kappa=_empty(3, 3))
        return {"kappa": kappa}
    g = kk.kald_phase_space(ctx, s[0], st.mesh, st.nu, st.opt, g=_empty(nq * nb))
    return {"g": _kept(g, st.case)}


def _phonon_outputs(nu, eig, vel):
    """What a phase-free comparison of phonons can use: the eigenvalues (nu |nu|;
    the acoustic nu at Gamma are square roots of rounding noise), the weight of
    every atom and direction in every mode, and the velocities; modes below
    omega_min, the translations at Gamma, carry no information and are zeroed."""
    live = (nu > NU_MIN)[..., None]
    return {"nu2": nu * nu.abs(), "weight": torch.where(live, eig.real ** 2 + eig.imag ** 2, 0.0),
            "vel": torch.where(live, vel, 0.0)}


# ---------------------------------------------------------------- work
def _fc3_blocks(case):
    return [len(_crystal("alloy" if "cells" in case else case["cell"], _cubic(n))[4])
            for n in (case["cells"].split(",") if "cells" in case else [case.get("size", "1")])]


def _n_atoms(case):
    if "cells" in case:
        return [4 * math.prod(_cubic(c)) for c in case["cells"].split(",")]
    return [{"ar": 1, "l11": 2}.get(case["cell"], 4 * math.prod(_cubic(case.get("size", "1"))))]


def work(case):
    """Each input read once and each output written once; floating operations of
    the projections of one momentum triple per orbit (1/12 of the ordered pairs),
    of the dense eigensolves and of the pair sums."""
    kind = case["kind"]
    nbs = [3 * n for n in _n_atoms(case)]
    nq = 1 if "cells" in case else math.prod(_ints(case["mesh"]))
    blocks = _fc3_blocks(case)
    vec = sum(nq * n * n for n in nbs) * 16
    modes = sum(nq * n for n in nbs) * 8
    fc = sum(b * 27 * 8 for b in blocks)
    fc2 = sum(79 * n // 3 * 72 for n in nbs)
    complex_flops = 1 if "cells" in case else 4
    pairs = 1.0 / 6.0 if "cells" in case else nq * nq / 12.0
    project = sum(pairs * n * (54.0 * b / 27 * 27 + 2 * 2 * complex_flops * float(n) ** 3) for n, b in zip(nbs, blocks))
    solve = sum(nq / (1.0 if "cells" in case else 2.0) * complex_flops * 8.0 * float(n) ** 3 for n in nbs)
    velocity = nq * nbs[0] * 79.0 * nbs[0] / 3 * 40
    qhgk = sum(3 * 2 * float(n) ** 3 / 2 for n in nbs)
    if kind == "kappa_rta":
        return {"bytes": vec + 2 * modes + fc2, "flops": velocity}
    if kind == "step":
        return {"bytes": vec + 2 * modes + fc + fc2, "flops": project + solve + velocity}
    if kind in ("linewidths", "linewidths_cells"):
        return {"bytes": vec + 2 * modes + fc, "flops": project}
    if kind == "phonons":
        return {"bytes": vec + 4 * modes + fc2, "flops": solve + velocity}
    if kind == "step_cells":
        return {"bytes": vec + 2 * modes + fc + fc2, "flops": project + solve + qhgk}
    if kind == "qhgk":
        return {"bytes": vec + 2 * modes + fc2, "flops": qhgk}
    if kind == "bte":
        return {"bytes": vec + modes + fc + 8.0 * (nq * nbs[0]) ** 2, "flops": 6 * project}
    return {"bytes": 2 * modes, "flops": nq * nq / 12.0 * float(nbs[0]) ** 3 * 20}


# ---------------------------------------------------------------- 64-bit results
def _occ(w, T):
    return torch.where(w > 0, 1.0 / torch.expm1(HBAR_EV_PS * w.clamp(min=1e-30) / (KB_EV * T)), 0.0)


def _shape(d, case):
    w = 2 * math.pi * case["sigma"]
    delta = case.get("delta", "gaussian")
    if delta == "gaussian":
        v = torch.exp(-0.5 * (d / w) ** 2) / (math.sqrt(2 * math.pi) * w)
    elif delta == "lorentzian":
        v = (w / math.pi) / (d * d + w * w)
    else:
        v = (1 - d.abs() / w).clamp(min=0.0) / w
    return torch.where(d.abs() < N_SIGMA * w, v, 0.0)


def _average(nu, g):
    """g averaged over chains of modes closer than DEGEN_TOL at one q (modes ascending)."""
    nu_h, out = nu.cpu().numpy(), g.cpu().numpy().copy()
    join = np.diff(nu_h, axis=1) < DEGEN_TOL
    for q in np.nonzero(join.any(axis=1))[0]:
        a = 0
        for b in range(1, nu_h.shape[1] + 1):
            if b == nu_h.shape[1] or not join[q, b - 1]:
                out[q, a:b] = out[q, a:b].mean()
                a = b
    return torch.as_tensor(out, device=g.device)


def _masked(nu):
    return torch.where(nu > NU_MIN, 2 * math.pi * nu, 0.0)


def _inv(w):
    return torch.where(w > 0, 1.0 / w.clamp(min=1e-30), 0.0)


def _weights(w, w1, w2, n1, n2, case):
    """The + and - energy weights, any broadcastable shapes (0 for masked modes)."""
    live = (w > 0) & (w1 > 0) & (w2 > 0)
    p = torch.where(live, (n1 - n2) * _shape(w + w1 - w2, case), 0.0)
    m = torch.where(live, 0.5 * (1 + n1 + n2) * _shape(w - w1 - w2, case), 0.0)
    return p, m


def _crystal_rates(s, mesh, nu, eig, case, visit):
    """For every q and chunk of q': visit(q, q' indices, q'' indices, |phi|^2 [q', s, s', s''], p, m)."""
    k = _fractions(mesh)
    nq, nb = nu.shape
    q = _qpoints(s, mesh)
    x = s.fc3_idx
    blk = s.fc3 / np.sqrt(s.masses[x[:, 0]] * s.masses[x[:, 1]] * s.masses[x[:, 5]])[:, None, None, None]
    a3 = np.arange(3)
    at = (((3 * x[:, 0, None] + a3)[:, :, None, None] * nb + (3 * x[:, 1, None] + a3)[:, None, :, None]) * nb +
          (3 * x[:, 5, None] + a3)[:, None, None, :])
    blk, at = _cuda(blk.reshape(-1, 27)), _cuda(at.reshape(-1))
    Rj, Rk = _cuda(x[:, 2:5] @ s.lattice), _cuda(x[:, 6:9] @ s.lattice)
    qd = _cuda(q)
    chi_j = torch.exp(-1j * (qd @ Rj.T))
    chi_k = torch.exp(-1j * (qd @ Rk.T))
    w, T = _masked(nu), case["T"]
    n = _occ(w, T)
    step = max(1, min((1 << 26) // max(nb ** 3, at.numel()), nq))
    for iq in range(nq):
        qpp = _flat(k[iq][None] + k, mesh)
        for c in range(0, nq, step):
            p_i = torch.arange(c, min(nq, c + step), device="cuda")
            pp = torch.as_tensor(qpp[c:c + step], device="cuda")
            ph = chi_j[p_i] * chi_k[pp].conj()
            W = torch.zeros((len(p_i), nb ** 3), dtype=torch.complex128, device="cuda")
            W.index_add_(1, at, (ph[:, :, None] * blk[None]).reshape(len(p_i), -1))
            Y = eig[iq] @ W.reshape(len(p_i), nb, nb * nb)                     # s, (b c)
            Y = Y.reshape(len(p_i), nb, nb, nb)
            Tm = torch.matmul(eig[p_i][:, None], Y)                            # s, s', c
            phi = torch.matmul(Tm, eig[pp].conj().transpose(-1, -2)[:, None])  # s, s', s''
            f2 = phi.real ** 2 + phi.imag ** 2
            gp, gm = _weights(w[iq][None, :, None, None], w[p_i][:, None, :, None], w[pp][:, None, None, :],
                              n[p_i][:, None, :, None], n[pp][:, None, None, :], case)
            visit(iq, p_i, pp, f2, gp, gm)


def _prefactor(nq):
    return HBAR_EV_PS * math.pi / 8.0 / nq * EV_A2_AMU ** 3


def _exact_gamma(s, mesh, nu, eig, case, average=True):
    nq, nb = nu.shape
    w = _masked(nu)
    iw = _inv(w)
    g = torch.zeros_like(nu)
    k = _fractions(mesh)

    def visit(iq, p, pp, f2, gp, gm):
        g[iq] += (f2 * (gp + gm) * iw[p][:, None, :, None] * iw[pp][:, None, None, :]).sum((0, 2, 3))

    _crystal_rates(s, mesh, nu, eig, case, visit)
    g = g * _prefactor(nq) * iw
    return _average(nu, g) if average else g


def _exact_gamma_only(s, nu, eig, case):
    E = eig[0].real.contiguous()
    nb = E.shape[0]
    x = s.fc3_idx
    blk = s.fc3 / np.sqrt(s.masses[x[:, 0]] * s.masses[x[:, 1]] * s.masses[x[:, 5]])[:, None, None, None]
    a3 = np.arange(3)
    at = _cuda(((3 * x[:, 1, None] + a3)[:, :, None] * nb + (3 * x[:, 5, None] + a3)[:, None, :]).reshape(-1))
    blk = _cuda(blk.reshape(-1, 3, 9))
    i3 = _cuda(3 * x[:, 0, None] + a3)
    w = _masked(nu[0])
    n, iw = _occ(w, case["T"]), _inv(w)
    g = torch.zeros_like(w)
    for mu in range(nb):
        if not float(w[mu]) > 0:
            continue
        Y = torch.zeros(nb * nb, dtype=torch.float64, device="cuda")
        Y.index_add_(0, at, (E[mu][i3][:, :, None] * blk).sum(1).reshape(-1))
        phi = E @ Y.reshape(nb, nb) @ E.T
        p, m = _weights(w[mu], w[:, None], w[None, :], n[:, None], n[None, :], case)
        g[mu] = (phi * phi * (p + m) * iw[:, None] * iw[None, :]).sum()
    return _average(nu, (g * _prefactor(1) * iw)[None])[0]


def _heat(w, T):
    x = HBAR_EV_PS * w.clamp(min=1e-30) / (KB_EV * T)
    return torch.where(w > 0, _KB * x * x * torch.exp(-x) / (1 - torch.exp(-x)) ** 2, 0.0)


def _velocity_matrices(s, mesh, nu, eig):
    """V [3][nq, nb, nb] (A/ps): eta_s^dagger dD/dq_a eta_s' / (2 sqrt(w w'))."""
    q, R = _qpoints(s, mesh), s.fc2_idx[:, 2:5] @ s.lattice
    w = _masked(nu)
    sc = torch.where((w[:, :, None] > 0) & (w[:, None, :] > 0),
                     EV_A2_AMU / (2 * torch.sqrt((w[:, :, None] * w[:, None, :]).clamp(min=1e-30))), 0.0)
    return [eig.conj() @ (-1j * _dynmat(s, q, R[:, a])) @ eig.transpose(-1, -2) * sc for a in range(3)]


def _volume(s):
    return abs(float(np.linalg.det(s.lattice)))


def _exact_rta(s, mesh, nu, eig, gamma, T):
    V = _velocity_matrices(s, mesh, nu, eig)
    w = _masked(nu)
    ok = (w > 0) & (gamma > 0)
    ct = torch.where(ok, _heat(w, T) / (2 * gamma.clamp(min=1e-300)), 0.0)
    ct = _average(nu, ct)
    ids = torch.cumsum(torch.cat([torch.zeros_like(nu[:, :1]),
                                  (torch.diff(nu, dim=1) >= DEGEN_TOL).to(nu.dtype)], 1), 1)
    same = (ids[:, :, None] == ids[:, None, :]) & ok[:, :, None] & ok[:, None, :]
    wt = torch.where(same, ct[:, :, None], 0.0)
    kap = torch.stack([torch.stack([(wt * (V[a] * V[b].conj()).real).sum() for b in range(3)]) for a in range(3)])
    return kap * 1e22 / (nu.shape[0] * _volume(s))


def _exact_qhgk(s, nu, eig, gamma, T):
    E = eig[0].real.contiguous()
    nb = E.shape[0]
    x = s.fc2_idx
    blk = s.fc2 / np.sqrt(s.masses[x[:, 0]] * s.masses[x[:, 1]])[:, None, None]
    dist = s.positions[x[:, 0]] - s.positions[x[:, 1]] - x[:, 2:5] @ s.lattice
    a3 = np.arange(3)
    at = _cuda(((3 * x[:, 0, None] + a3)[:, :, None] * nb + (3 * x[:, 1, None] + a3)[:, None, :]).reshape(-1))
    w = _masked(nu[0])
    ok = (w > 0) & (gamma > 0)
    sq = torch.where(ok, torch.sqrt(_inv(w)), 0.0)
    W = []
    for a in range(3):
        A = torch.zeros(nb * nb, dtype=torch.float64, device="cuda")
        A.index_add_(0, at, _cuda((blk * dist[:, a, None, None]).reshape(-1)))
        W.append(E @ A.reshape(nb, nb) @ E.T * sq[:, None] * sq[None, :] * (0.5 * EV_A2_AMU))
    n, c = _occ(w, T), _heat(w, T)
    dw = w[:, None] - w[None, :]
    near = dw.abs() < 2 * math.pi * DEGEN_TOL
    cc = torch.where(near, 0.5 * (c[:, None] + c[None, :]),
                     _HBAR * 1e12 * w[:, None] * w[None, :] / T * (n[None, :] - n[:, None]) /
                     torch.where(near, 1.0, dw))
    gs = gamma[:, None] + gamma[None, :]
    wt = torch.where(ok[:, None] & ok[None, :], cc * gs / (dw * dw + gs * gs).clamp(min=1e-300), 0.0)
    kap = torch.stack([torch.stack([(wt * W[a] * W[b]).sum() for b in range(3)]) for a in range(3)])
    return kap * 1e22 / _volume(s)


def _exact_bte(s, mesh, nu, eig, case):
    nq, nb = nu.shape
    k, w = _fractions(mesh), _masked(nu)
    iw = _inv(w)
    neg = torch.as_tensor(_flat(-k, mesh), device="cuda")
    N = nq * nb
    g0 = torch.zeros_like(nu)
    G1 = torch.zeros((nq, nb, nq, nb), dtype=torch.float64, device="cuda")

    def visit(iq, p, pp, f2, gp, gm):
        i1, i2 = iw[p][:, None, :, None], iw[pp][:, None, None, :]
        g0[iq] += (f2 * (gp + gm) * i1 * i2).sum((0, 2, 3))
        G1[iq].index_add_(1, p, (f2 * gp * i2).sum(3).transpose(0, 1))
        G1[iq].index_add_(1, neg[p], -(f2 * gm * i2).sum(3).transpose(0, 1))
        G1[iq].index_add_(1, pp, -(f2 * (gp + gm) * i1).sum(2).transpose(0, 1))

    _crystal_rates(s, mesh, nu, eig, case, visit)
    g0 = (g0 * _prefactor(nq) * iw).reshape(-1)
    G1 = (G1 * (_prefactor(nq) * iw * iw)[:, :, None, None]).reshape(N, N)
    V = _velocity_matrices(s, mesh, nu, eig)
    v = torch.stack([torch.diagonal(x, dim1=1, dim2=2).real.reshape(-1) for x in V], 1)
    ok = (w.reshape(-1) > 0) & (g0 > 0)
    A = 2 * (torch.diag(g0) + G1)
    A = torch.where(ok[:, None] & ok[None, :], A, torch.eye(N, dtype=A.dtype, device=A.device))
    lam = torch.linalg.solve(A, torch.where(ok[:, None], v, 0.0))
    c = torch.where(ok, _heat(w.reshape(-1), case["T"]), 0.0)
    return (v * c[:, None]).T @ lam * 1e22 / (nq * _volume(s))


def _exact_phase_space(mesh, nu, case):
    nq, nb = nu.shape
    k, w = _fractions(mesh), _masked(nu)
    n = _occ(w, case["T"])
    g = torch.zeros_like(nu)
    step = max(1, (1 << 25) // nb ** 3)
    for iq in range(nq):
        qpp = _flat(k[iq][None] + k, mesh)
        for c in range(0, nq, step):
            p, pp = torch.arange(c, min(nq, c + step), device="cuda"), torch.as_tensor(qpp[c:c + step], device="cuda")
            gp, gm = _weights(w[iq][None, :, None, None], w[p][:, None, :, None], w[pp][:, None, None, :],
                              n[p][:, None, :, None], n[pp][:, None, None, :], case)
            g[iq] += (gp + gm).sum((0, 2, 3))
    return g / nq


def exact(case, seed):
    kind = case["kind"]
    nbs = [3 * n for n in _n_atoms(case)]
    mesh = (1, 1, 1) if "cells" in case else tuple(_ints(case["mesh"]))
    nq = math.prod(mesh)
    # projections of all ordered pairs, in 64 bits, within a few seconds
    pairs_ok = nq * nq * (float(nbs[0]) ** 4 + 3e5) < 5e11
    if kind in ("linewidths", "bte") and not pairs_ok:
        return None
    if kind == "linewidths_cells" and max(nbs) > 800:
        return None
    if kind == "phase_space" and nq * nq * float(nbs[0]) ** 3 > 2e10:
        return None
    systems = _systems(case, seed)
    ph = [_phonons(s, mesh) for s in systems]
    (nu, eig), s = ph[0], systems[0]
    if kind == "kappa_rta":
        gamma = _average(nu, _model_gamma(nu.reshape(-1), seed).reshape(nq, -1))
        return {"kappa": _exact_rta(s, mesh, nu, eig, gamma, case["T"])}
    if kind == "step":
        out = {"nu2": nu * nu.abs(), "gamma": None, "kappa": None}
        if pairs_ok:
            g = _exact_gamma(s, mesh, nu, eig, case)
            out.update(gamma=g.reshape(-1), kappa=_exact_rta(s, mesh, nu, eig, g, case["T"]))
        return out
    if kind == "linewidths":
        return {"gamma": _exact_gamma(s, mesh, nu, eig, case).reshape(-1), "triplets": None}
    if kind == "phonons":
        V = _velocity_matrices(s, mesh, nu, eig)
        v = torch.stack([torch.diagonal(x, dim1=1, dim2=2).real for x in V], -1)
        return _phonon_outputs(nu, eig, v)
    if kind in ("linewidths_cells", "step_cells"):
        small = max(nbs) <= 800 and sum(float(n) ** 4 for n in nbs) < 2e12
        g = [_exact_gamma_only(x, *p, case) for x, p in zip(systems, ph)] if small else None
        gamma = torch.cat(g) if small else None
        if kind == "linewidths_cells":
            return {"gamma": gamma, "triplets": None}
        nu2 = torch.cat([(p[0] * p[0].abs()).reshape(-1) for p in ph])
        kap = torch.stack([_exact_qhgk(x, *p, y, case["T"]) for x, p, y in zip(systems, ph, g)]) if small else None
        return {"nu2": nu2, "gamma": gamma, "kappa": kap}
    if kind == "qhgk":
        g = torch.split(_model_gamma(torch.cat([p[0].reshape(-1) for p in ph]), seed), nbs)
        return {"kappa": torch.stack([_exact_qhgk(x, *p, y, case["T"]) for x, p, y in zip(systems, ph, g)])}
    if kind == "bte":
        return {"kappa": _exact_bte(s, mesh, nu, eig, case)}
    return {"g": _exact_phase_space(mesh, nu, case).reshape(-1)}
