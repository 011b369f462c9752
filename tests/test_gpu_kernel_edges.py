"""Edge sizes of individual kernels (GPU), against the FP64 oracle or the
library's own FP64 path, which other tests hold to the oracle at 1e-10.

Tolerances are those of the modes: 1e-5 of gamma for the FP32 and BF16-split
linewidths (the energy windows and weights are FP32 in both), 1e-10 for FP64
results."""

import numpy as np
import pytest

import kald_inputs as ki
from oracle import phonons as ph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def k():
    from paper_2009_01967_gb300 import build
    build.build()
    import paper_2009_01967_gb300 as kk
    ctx = kk.Context(0)
    yield kk, ctx
    ctx.close()


def _rel(a, b):
    return np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-6 * np.abs(b).max()))


@pytest.mark.parametrize("cell,extra", [((3, 3, 1), 0), ((9, 1, 1), 0), ((5, 2, 1), 0), ((3, 3, 1), 300)])
def test_gamma_only_y_build(k, cell, extra):
    """108, 108 and 120 modes (a last batch of 12, 12 and 24 of 32 modes, no
    whole 32-mode tile of eigenvector pairs at the end); 300 random blocks add
    groups of every length up to the warp-per-group limit and a Phi3 without
    symmetry."""
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=5)
    if extra:
        s = ki.random_fc3_system(s, extra, seed=3)
    nu, eig = ph.phonons(s, (1, 1, 1))
    out = {}
    for prec in ("fp64", "bf16split"):
        opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=prec)
        out[prec] = kk.kald_linewidths(ctx, [s], (1, 1, 1), nu.ravel(), eig.ravel(), opt)
    assert abs(out["fp64"][1][1] - out["bf16split"][1][1]) <= 1e-5 * out["fp64"][1][1]
    assert _rel(out["bf16split"][0], out["fp64"][0]) < 1e-5


@pytest.mark.parametrize("mesh,extra,cap", [((1, 1, 1), 40, 0), ((7, 2, 3), 40, 0), ((9, 5, 1), 0, 0),
                                            ((4, 4, 4), 40, 1 << 20)])
def test_register_kernel_phase_tables(k, mesh, extra, cap):
    """Phase sums from the per-q tables: a single q-point, uneven meshes with a
    last partial pass over the q', random blocks with two different cell
    vectors (summed per pair), and no tables at all under a workspace cap that
    they would not fit."""
    from oracle import anharmonic as an
    kk, ctx = k
    w = ki.small_binary(mesh=mesh, sigma=0.1)
    s = ki.random_fc3_system(w.systems[0], extra, seed=7) if extra else w.systems[0]
    nu, eig = ph.phonons(s, mesh)
    g_o = an.linewidths(s, mesh, nu, eig, w.T, w.sigma_thz, w.n_sigma)
    ctx.set_workspace_limit(cap)
    try:
        for prec, tol in (("fp64", 1e-10), ("fp32", 1e-5)):
            opt = kk.Options(temperature_K=w.T, sigma_thz=w.sigma_thz, n_sigma=w.n_sigma, precision=prec)
            g, _ = kk.kald_linewidths(ctx, s, mesh, nu, eig, opt)
            assert _rel(g.reshape(g_o.shape), g_o) < tol
    finally:
        ctx.set_workspace_limit(0)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("nb,mesh,sigma", [(3, (2, 3, 1), 0.3), (5, (3, 1, 1), 5.0), (130, (2, 1, 1), 0.02)])
def test_phase_space_sliding_windows(k, nb, mesh, sigma, precision, tol):
    """Frequencies in no order, with equal, negative and masked ones, windows
    wider than the spectrum and narrow ones, more modes than one CTA's threads."""
    from types import SimpleNamespace
    from oracle import anharmonic as an
    kk, ctx = k
    if nb % 3:
        nb += 3 - nb % 3
    rng = np.random.default_rng(nb)
    nq = int(np.prod(mesh))
    nu = rng.uniform(0.2, 2.0, (nq, nb))
    nu[:, nb // 2] = nu[:, 0]
    nu[0, 1], nu[-1, 0] = -0.3, 0.001
    s = ki.small_binary(mesh=mesh).systems[0]
    n = nb // 3
    s = SimpleNamespace(masses=np.full(n, 20.0), positions=np.arange(3.0 * n).reshape(n, 3), lattice=10 * np.eye(3),
                        fc2_idx=s.fc2_idx[:0], fc2=s.fc2[:0], fc3_idx=s.fc3_idx[:0], fc3=s.fc3[:0])
    g_o = an.phase_space(mesh, nu, 300.0, sigma, 3.0)
    opt = kk.Options(temperature_K=300.0, sigma_thz=sigma, precision=precision)
    g = kk.kald_phase_space(ctx, s, mesh, nu, opt).reshape(g_o.shape)
    assert np.all(g[nu <= 0.01] == 0.0)
    # the oracle's - process takes w(-q'); on this spectrum, which is not that of
    # a crystal, it is compared on meshes where -q' = q' or with nu made even
    neg = np.array([np.ravel_multi_index(tuple((-np.array(np.unravel_index(q, mesh))) % mesh), mesh) for q in range(nq)])
    if np.any(neg != np.arange(nq)):
        nu = np.where((neg < np.arange(nq))[:, None], nu[neg], nu)
        g_o = an.phase_space(mesh, nu, 300.0, sigma, 3.0)
        g = kk.kald_phase_space(ctx, s, mesh, nu, opt).reshape(g_o.shape)
    assert _rel(g, g_o) < tol


@pytest.mark.parametrize("cell,mesh", [("binary", (3, 2, 2)), ("fcc4", (2, 2, 3)), ("fcc20", (3, 1, 1))])
@pytest.mark.parametrize("asym", [0.0, 0.05])
def test_kappa_rta_from_diagonal_elements(k, cell, mesh, asym):
    """Two, four and 20 atoms (meshes with q-points off the zone boundary, where
    velocities do not vanish by time reversal): degenerate sets (the off-diagonal elements), a
    Phi2 without the (i, j) <-> (j, i) symmetry (complex diagonal elements, an
    atom pair listed in one order only), and eigenvectors at -q that are not the
    conjugates of those at q."""
    from dataclasses import replace
    from oracle import conductivity as co
    kk, ctx = k
    s = ki.small_binary(mesh=mesh).systems[0] if cell == "binary" else \
        ki.fcc_supercell_system(1 if cell == "fcc4" else (5, 1, 1), seed=7)
    nu, eig = ph.phonons(s, mesh)
    rng = np.random.default_rng(3)
    eig = eig * np.exp(2j * np.pi * rng.random(nu.shape))[..., None]
    g = np.where(nu > 0.01, 0.1 + 0.02 * nu ** 2, 0.0)
    if asym:
        fc2 = s.fc2 * (1.0 + asym * rng.standard_normal(s.fc2.shape))
        keep = ~((s.fc2_idx[:, 0] == 1) & (s.fc2_idx[:, 1] == 0))
        s = replace(s, fc2=fc2[keep], fc2_idx=s.fc2_idx[keep])
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)
    kap = kk.kald_kappa_rta(ctx, s, mesh, nu, eig, g, opt)
    if asym:
        # (the oracle symmetrises dD/dq: the general kernel of the call without
        # scratch, which runs over every block for every pair of modes)
        torch = pytest.importorskip("torch")
        dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (nu, eig, g)]
        out = torch.zeros((3, 3), dtype=torch.float64, device="cuda")
        kap_o = kk.kald_kappa_rta_noalloc(ctx, s, mesh, *dev, opt, out).cpu().numpy()
    else:
        kap_o = co.kappa_rta(s, mesh, nu, eig, g, 300.0)
    np.testing.assert_allclose(kap, kap_o, rtol=1e-10, atol=1e-10 * np.abs(kap_o).max())


def _qhgk_system(cell, asym):
    from dataclasses import replace
    s = ki.fcc_supercell_system(cell, seed=5)
    if asym:
        rng = np.random.default_rng(3)
        s = replace(s, fc2=s.fc2 * (1.0 + 0.05 * rng.standard_normal(s.fc2.shape)))
    return s


@pytest.mark.parametrize("cell,asym", [(1, False), (2, True), ((3, 3, 1), False), ((13, 1, 1), True), ((11, 2, 2), False)])
def test_generalised_velocities_exact_product(k, cell, asym):
    """12, 96, 108, 156 and 528 modes (less than a tile, a remainder of one column
    half, one chunk of 512 and a remainder), antisymmetric (the upper tiles and
    their mirror image) and not (a Phi2 without the pair symmetry): W against
    FP64 NumPy to 1e-13 of its largest element, kappa to 1e-10."""
    from oracle import conductivity as co
    kk, ctx = k
    s = _qhgk_system(cell, asym)
    nb = s.n_branches
    rng = np.random.default_rng(nb)
    # any orthonormal real vectors will do; one row with a wide range of magnitudes
    E = np.linalg.qr(rng.standard_normal((nb, nb)))[0]
    E[0] = np.exp(rng.uniform(-60, 0, nb))
    eig = E.astype(np.complex128)[None]
    nu = np.sort(rng.uniform(0.1, 2.0, (1, nb)))
    g = 0.05 + 0.02 * rng.random(nb)
    W_o = co.generalized_velocity(s, nu, eig)
    kap_o = co.kappa_qhgk(s, nu, eig, g, 300.0, W=W_o)
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)
    kap, W = kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt, want_vgen=True)
    if cell == 1:                                  # W vanishes by symmetry in the cubic 4-atom cell
        assert np.abs(W).max() < 1e-13 and np.abs(kap).max() < 1e-25
    else:
        np.testing.assert_allclose(W, W_o, rtol=0, atol=1e-13 * np.abs(W_o).max())
        np.testing.assert_allclose(kap[0], kap_o, rtol=1e-10, atol=1e-10 * np.abs(kap_o).max())
    kap2, _ = kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt)
    np.testing.assert_array_equal(kap2, kap)
    D = kk.kald_diffusivity(ctx, [s], nu.ravel(), eig.ravel(), g, opt)
    gs = g[:, None] + g[None, :]
    tau = gs / ((2 * np.pi * (nu.T - nu)) ** 2 + gs ** 2)
    D_o = (W_o ** 2 * tau[None]).sum(axis=(0, 2)) / 3
    if cell != 1:
        np.testing.assert_allclose(D, D_o, rtol=1e-10, atol=1e-12 * D_o.max())


def test_generalised_velocities_wait_limit(k):
    """A wait that runs out in the product is reported, and the context goes on."""
    kk, ctx = k
    s = ki.fcc_supercell_system((3, 3, 1), seed=5)
    nu, eig = ph.phonons(s, (1, 1, 1))
    g = np.where(nu > 0.01, 0.1, 0.0).ravel()
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)
    ref, _ = kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt)
    ctx.set_wait_limit(1)
    try:
        with pytest.raises(kk.KaldError) as e:
            kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt)
        assert e.value.status == 5
    finally:
        ctx.set_wait_limit(0)
    kap, _ = kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt)
    np.testing.assert_array_equal(kap, ref)


def _springs(n, kind):
    """A Gamma-only n-atom system whose 3n x 3n dynamical matrix (masses 1) is a
    given symmetric matrix: clustered, multiple and split spectra."""
    from types import SimpleNamespace
    nb = 3 * n
    rng = np.random.default_rng(n)
    Q = np.linalg.qr(rng.standard_normal((nb, nb)))[0]
    lam = {"spread": np.linspace(0.1, 4.0, nb),
           "multiple": np.repeat([0.5, 1.0, 1.0 + 1e-13, 3.0], (nb + 3) // 4)[:nb],
           "clustered": 1.0 + 1e-9 * np.arange(nb) + (np.arange(nb) % 3),
           "zero": np.zeros(nb)}.get(kind)
    D = np.diag(np.arange(1.0, nb + 1) / nb) if kind == "diagonal" else (Q * lam) @ Q.T
    D = 0.5 * (D + D.T)
    idx = np.array([[i, j, 0, 0, 0] for i in range(n) for j in range(n)], np.int32)
    fc2 = np.array([D[3 * i:3 * i + 3, 3 * j:3 * j + 3] for i in range(n) for j in range(n)])
    s = SimpleNamespace(masses=np.ones(n), positions=rng.random((n, 3)), lattice=10 * np.eye(3), fc2_idx=idx, fc2=fc2,
                        fc3_idx=np.zeros((0, 9), np.int32), fc3=np.zeros((0, 3, 3, 3)))
    return s, D


@pytest.mark.parametrize("n", [1, 5, 6, 11, 21, 32])
@pytest.mark.parametrize("kind", ["spread", "multiple", "clustered", "zero", "diagonal"])
def test_hermitian_eigensolver_spectra(k, n, kind):
    """3 to 96 branches (QL below 16, inverse iteration above, 15, 18, 33, 63 and
    96 rows): well separated, multiple and clustered eigenvalues, a zero and a
    diagonal matrix (no reflector, T split everywhere).  Eigenvalues, residuals
    and orthonormality to 1e-13 of |D| and of one."""
    from oracle.units import EV_A2_AMU
    kk, ctx = k
    s, D = _springs(n, kind)
    nu, eig, _ = kk.kald_phonons(ctx, s, (1, 1, 1), want_vel=False)
    E = eig[0].T                                            # columns = modes
    scale = max(np.abs(D).sum(axis=1).max(), 1e-30)
    lam = np.sign(nu[0]) * (2 * np.pi * nu[0]) ** 2 / EV_A2_AMU
    np.testing.assert_allclose(lam, np.linalg.eigvalsh(D), rtol=0, atol=1e-13 * scale)
    np.testing.assert_allclose(E.conj().T @ E, np.eye(3 * n), rtol=0, atol=1e-13)
    assert np.abs(D @ E - E * lam).max() <= 1e-13 * scale


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("cell,mesh,extra,cap", [((1, 1, 1), (3, 4, 2), 0, 0), ((1, 1, 1), (2, 2, 1), 80, 0),
                                                 ((2, 1, 1), (3, 3, 1), 0, 0), ((3, 1, 1), (2, 1, 2), 0, 1 << 23),
                                                 ((5, 1, 1), (2, 1, 1), 60, 0)])
def test_cuda_core_kernel_orbits_and_tables(k, cell, mesh, extra, cap, precision, tol):
    """Four to 20 atoms (12 to 60 branches): one projection per orbit of momentum
    triples for a symmetric Phi3, every pair for one with random blocks (their own
    phase class), no tables under a workspace cap; the same sums and the same
    delta-allowed count with no symmetry at all."""
    from oracle import anharmonic as an
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=7)
    if extra:
        s = ki.random_fc3_system(s, extra, seed=9)
    nu, eig = ph.phonons(s, mesh)
    g_o = an.linewidths(s, mesh, nu, eig, 300.0, 0.1, 3.0)
    count = {}
    ctx.set_workspace_limit(cap)
    try:
        for sym in ("all", "inversion", "none"):
            opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=precision, symmetry=sym)
            g, count[sym] = kk.kald_linewidths(ctx, s, mesh, nu, eig, opt)
            assert _rel(g.reshape(g_o.shape), g_o) < tol
    finally:
        ctx.set_workspace_limit(0)
    assert count["all"] == count["inversion"] == count["none"]


@pytest.mark.parametrize("cell,mesh,extra,tables", [((5, 5, 1), (2, 1, 1), 0, True), ((5, 5, 1), (3, 1, 2), 3000, True),
                                                    ((23, 1, 1), (1, 3, 1), 40, True), ((4, 2, 3), (2, 2, 1), 40, True),
                                                    ((4, 4, 2), (2, 1, 1), 0, False), ((4, 4, 2), (2, 1, 1), 40, False),
                                                    ((4, 4, 2), (1, 1, 1), 0, True)])
def test_tensor_core_gather(k, cell, mesh, extra, tables):
    """The phase sum of the BF16-split crystal path for 69, 72, 75 (odd rows) and 96
    branches: terms of all classes, random blocks (alone and several per atom
    triple), one q-point, and no tables at the smallest workspace the call takes;
    gamma and the delta-allowed count against the FP64 mode."""
    from kald_inputs.configs import A_FCC
    from kald_inputs.lattice import fcc_primitive
    from kald_inputs.lj import lj_system
    kk, ctx = k
    lat = fcc_primitive(A_FCC)[0]
    at = np.array(list(np.ndindex(*cell)))
    s = lj_system(lat * np.array(cell)[:, None], at @ lat, np.where(np.arange(len(at)) % 3 == 1, 60.0, 39.948))
    if extra:
        s = ki.random_fc3_system(s, extra, seed=4)
    nu, eig = ph.phonons(s, mesh)
    opt = {p: kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=p) for p in ("fp64", "bf16split")}
    ref, cnt = kk.kald_linewidths(ctx, [s], mesh, nu.ravel(), eig.ravel(), opt["fp64"])
    if not tables:
        ctx.set_workspace_limit(_smallest_workspace(kk, ctx, s, mesh, nu, eig, opt["bf16split"]))
    try:
        got, cnt2 = kk.kald_linewidths(ctx, [s], mesh, nu.ravel(), eig.ravel(), opt["bf16split"])
    finally:
        ctx.set_workspace_limit(0)
    assert abs(cnt[1] - cnt2[1]) <= 1e-5 * cnt[1]
    assert _rel(got, ref) < 1e-5


def _smallest_workspace(kk, ctx, s, mesh, nu, eig, opt):
    """Bytes the call asks for when it cannot have what it would like."""
    import re
    ctx.set_workspace_limit(1)
    try:
        with pytest.raises(kk.KaldError) as e:
            kk.kald_linewidths(ctx, [s], mesh, nu.ravel(), eig.ravel(), opt)
        return int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    finally:
        ctx.set_workspace_limit(0)


@pytest.mark.parametrize("cell,mesh,precision", [((1, 1, 1), (3, 3, 2), "fp64"), ((2, 1, 1), (2, 3, 1), "fp32"),
                                                 (None, (5, 5, 4), "fp64"), (None, (5, 5, 4), "fp32")])
def test_linewidths_at_the_smallest_workspace(k, cell, mesh, precision):
    """Under a workspace cap at which the tables or the orbits do not fit, the call
    does without them and gives the same linewidths and count."""
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=7) if cell else ki.small_binary().systems[0]
    nu, eig = ph.phonons(s, mesh)
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=precision)
    ref, cnt = kk.kald_linewidths(ctx, [s], mesh, nu.ravel(), eig.ravel(), opt)
    least = _smallest_workspace(kk, ctx, s, mesh, nu, eig, opt)
    for cap in (least, least + least // 8, 2 * least):
        ctx.set_workspace_limit(cap)
        try:
            got, cnt2 = kk.kald_linewidths(ctx, [s], mesh, nu.ravel(), eig.ravel(), opt)
        finally:
            ctx.set_workspace_limit(0)
        assert list(cnt) == list(cnt2)
        assert _rel(got, ref) < (1e-10 if precision == "fp64" else 1e-5)


def test_batch_plans_equal_single_calls(k):
    """A batch whose systems repeat, some hashed on several threads (more than a
    megabyte of force constants), gives what each system gives alone, from new and
    from kept plans; a faulty system in it is refused with its own message."""
    kk, ctx = k
    big, small = ki.fcc_supercell_system((4, 4, 3), seed=1), ki.fcc_supercell_system((3, 3, 1), seed=2)
    systems = [small, big, ki.random_fc3_system(small, 30, seed=3), big, small]
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision="bf16split")
    ph1 = [ph.phonons(s, (1, 1, 1)) for s in (big, small)]
    by = [1, 0, 1, 0, 1]
    nu, eig = (np.concatenate([ph1[b][c].ravel() for b in by]) for c in (0, 1))
    with kk.Context(0) as fresh:
        runs = [kk.kald_linewidths(fresh, systems, (1, 1, 1), nu, eig, opt) for _ in range(2)]
    alone = [kk.kald_linewidths(ctx, [s], (1, 1, 1), ph1[b][0].ravel(), ph1[b][1].ravel(), opt)
             for s, b in zip(systems, by)]
    for g, cnt in runs:
        np.testing.assert_array_equal(np.asarray(g).ravel(), np.concatenate([np.asarray(a[0]).ravel() for a in alone]))
        assert cnt[1] == sum(a[1][1] for a in alone)
    bad = ki.fcc_supercell_system((3, 3, 1), seed=2)
    bad.fc3_idx[5, 0] = bad.n_atoms
    nu3, eig3 = (np.tile(ph1[1][c].ravel(), 3) for c in (0, 1))
    with pytest.raises(kk.KaldError, match="fc3_idx"):
        kk.kald_linewidths(ctx, [small, bad, small], (1, 1, 1), nu3, eig3, opt)


@pytest.mark.parametrize("cell,sigma,shape", [((3, 3, 1), 0.02, "gaussian"), ((3, 3, 2), 0.2, "gaussian"),
                                              ((4, 3, 3), 0.05, "gaussian"), ((4, 3, 3), 0.02, "lorentzian"),
                                              ((5, 2, 1), 0.1, "triangular")])
def test_gamma_only_triples_projected_once(k, cell, sigma, shape):
    """108 to 432 modes (one to four tiles, the last one partial), windows narrower
    and wider than half the lowest frequencies: each unordered triple of modes
    projected once gives the linewidths and the exact count of one projection per
    ordered triple, at the usual workspace and at the smallest."""
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=11)
    nu, eig = ph.phonons(s, (1, 1, 1))
    def run(**o):
        opt = kk.Options(temperature_K=300.0, sigma_thz=sigma, delta=shape, **o)
        return kk.kald_linewidths(ctx, [s], (1, 1, 1), nu.ravel(), eig.ravel(), opt)
    ref, _ = run(precision="fp64")
    each, count = run(precision="bf16split", symmetry="inversion")
    once, count1 = run(precision="bf16split")
    least = _smallest_workspace(kk, ctx, s, (1, 1, 1), nu, eig,
                                kk.Options(temperature_K=300.0, sigma_thz=sigma, delta=shape, precision="bf16split"))
    ctx.set_workspace_limit(least)
    try:
        small, count2 = run(precision="bf16split")
    finally:
        ctx.set_workspace_limit(0)
    assert tuple(count) == tuple(count1) == tuple(count2)
    for g in (each, once, small):
        assert _rel(g, ref) < 1e-5


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("atoms,mesh,sigma", [(2, (2, 1, 1), 0.2), (2, (3, 3, 3), 0.1), (2, (5, 4, 2), 0.05),
                                              (1, (4, 4, 4), 0.2), (1, (7, 3, 1), 0.1)])
def test_register_kernel_orbits(k, atoms, mesh, sigma, precision, tol):
    """One- and two-atom cells, meshes with and without self-inverse and 3 q = 0
    points, fewer and more orbits than a pass holds: one projection per orbit gives
    the linewidths of the oracle and the exact count of one projection per pair."""
    from oracle import anharmonic as an
    kk, ctx = k
    w = ki.small_binary(mesh=mesh, sigma=sigma) if atoms == 2 else ki.small_fcc_prim(mesh=mesh, sigma=sigma)
    s = w.systems[0]
    nu, eig = ph.phonons(s, mesh)
    g_o = an.linewidths(s, mesh, nu, eig, w.T, sigma, 3.0)
    count = {}
    for sym in ("all", "inversion", "none"):
        opt = kk.Options(temperature_K=w.T, sigma_thz=sigma, precision=precision, symmetry=sym)
        g, count[sym] = kk.kald_linewidths(ctx, s, mesh, nu, eig, opt)
        assert _rel(g.reshape(g_o.shape), g_o) < tol
    assert count["all"] == count["inversion"] == count["none"]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("mesh", [(4, 3, 2), (1, 5, 1)])
@pytest.mark.parametrize("change", [0.0, 1e-14, 1e-3])
def test_phase_space_of_mirrored_frequencies(k, mesh, change, precision):
    """Frequencies of -q equal to those of q, to rounding, or not: the sums of one
    q-point of each pair, or of both, are those of the smallest workspace, where
    every q-point is summed by itself (1e-10: 4e-13 of the largest frequency moves a
    Gaussian weight by 3 w_max / sigma times that; FP32 1e-5 of the mode)."""
    import re
    kk, ctx = k
    s = ki.small_binary(mesh=mesh).systems[0]
    nq, nb = int(np.prod(mesh)), 6
    rng = np.random.default_rng(3)
    nu = rng.uniform(0.3, 2.0, (nq, nb))
    neg = np.array([np.ravel_multi_index(tuple((-np.array(np.unravel_index(q, mesh))) % mesh), mesh) for q in range(nq)])
    nu = np.where((neg < np.arange(nq))[:, None], nu[neg], nu)
    last = int(np.flatnonzero(neg < np.arange(nq))[-1])
    nu[last, 3] *= 1.0 + change
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.05, precision=precision)
    g = kk.kald_phase_space(ctx, s, mesh, nu, opt)
    ctx.set_workspace_limit(1)
    try:
        with pytest.raises(kk.KaldError) as e:
            kk.kald_phase_space(ctx, s, mesh, nu, opt)
        ctx.set_workspace_limit(int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)))
        ref = kk.kald_phase_space(ctx, s, mesh, nu, opt)
    finally:
        ctx.set_workspace_limit(0)
    assert np.max(np.abs(g - ref)) <= (1e-10 if precision == "fp64" else 1e-5) * np.max(np.abs(ref))
    assert np.all(np.asarray(ref) > 0)


@pytest.mark.parametrize("cell,mesh", [((1, 1, 1), (3, 4, 2)), ((2, 2, 2), (2, 1, 1)), ((2, 1, 1), (1, 1, 1)),
                                       (None, (5, 3, 1))])
def test_phonons_and_conductivity_at_the_smallest_workspace(k, cell, mesh):
    """The eigensolver in batches, the velocities' table and the mirrored velocities in
    the matrices' place, the conductivity without stored velocities: what a call gives
    with the workspace it would like (one- to 32-atom cells, meshes with and without
    mirrored points)."""
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=7) if cell else ki.small_binary().systems[0]
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)

    def least(f):
        import re
        ctx.set_workspace_limit(1)
        with pytest.raises(kk.KaldError) as e:
            f()
        ctx.set_workspace_limit(int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)))

    try:
        nu, eig, vel = kk.kald_phonons(ctx, s, mesh)
        least(lambda: kk.kald_phonons(ctx, s, mesh))
        nu2, eig2, vel2 = kk.kald_phonons(ctx, s, mesh)
        np.testing.assert_array_equal(nu, nu2)
        np.testing.assert_array_equal(eig, eig2)
        np.testing.assert_array_equal(vel, vel2)
        ctx.set_workspace_limit(0)
        g = np.where(nu > 0.01, 0.1, 0.0).ravel()
        kappa = kk.kald_kappa_rta(ctx, s, mesh, nu, eig, g, opt)
        least(lambda: kk.kald_kappa_rta(ctx, s, mesh, nu, eig, g, opt))
        kappa2 = kk.kald_kappa_rta(ctx, s, mesh, nu, eig, g, opt)
    finally:
        ctx.set_workspace_limit(0)
    np.testing.assert_allclose(kappa2, kappa, rtol=1e-9, atol=1e-11 * np.abs(kappa).max() + 1e-30)


@pytest.mark.parametrize("cell", [(3, 3, 1), (4, 4, 2)])
def test_generalised_velocities_one_direction_at_a_time(k, cell):
    """108 and 384 modes: one direction's slices at a time, bit for bit."""
    import re
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=5)
    nu, eig = ph.phonons(s, (1, 1, 1))
    g = np.where(nu > 0.01, 0.1, 0.0).ravel()
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)
    for call in (lambda: kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), g, opt)[0],
                 lambda: kk.kald_diffusivity(ctx, [s], nu.ravel(), eig.ravel(), g, opt)):
        ref = call()
        ctx.set_workspace_limit(1)
        try:
            with pytest.raises(kk.KaldError) as e:
                call()
            ctx.set_workspace_limit(int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)))
            got = call()
        finally:
            ctx.set_workspace_limit(0)
        np.testing.assert_array_equal(got, ref)


def test_more_systems_than_are_planned_at_once(k):
    """66 Gamma-only systems (64 are planned together), small cells around a large one:
    the linewidths of each alone, bit for bit."""
    kk, ctx = k
    small = [ki.fcc_supercell_system((1, 1, 1), seed=i) for i in range(3)]
    big = ki.fcc_supercell_system((3, 3, 1), seed=9)
    systems = [small[i % 3] for i in range(65)]
    systems.insert(40, big)
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.2, precision="bf16split")
    ph1 = {id(s): ph.phonons(s, (1, 1, 1)) for s in small + [big]}
    alone = {id(s): kk.kald_linewidths(ctx, [s], (1, 1, 1), ph1[id(s)][0].ravel(), ph1[id(s)][1].ravel(), opt)[0]
             for s in small + [big]}
    nu, eig = (np.concatenate([ph1[id(s)][c].ravel() for s in systems]) for c in (0, 1))
    got, _ = kk.kald_linewidths(ctx, systems, (1, 1, 1), nu, eig, opt)
    np.testing.assert_array_equal(got, np.concatenate([np.asarray(alone[id(s)]).ravel() for s in systems]))


@pytest.mark.parametrize("cell,mesh,precision", [(None, (3, 3, 3), "fp64"), (None, (3, 3, 3), "fp32"),
                                                 ((1, 1, 1), (3, 2, 2), "fp64"), ((2, 2, 2), (2, 1, 1), "bf16split"),
                                                 ((3, 3, 1), (1, 1, 1), "bf16split")])
def test_repeated_blocks_are_added(k, cell, mesh, precision):
    """A Phi3 block listed twice counts twice, so that Phi3 is not symmetric under
    permutations although every single block has its partners: the linewidths are
    those of the same Phi3 with the two blocks added into one, which no symmetry check
    takes for symmetric (two, four and 32 atoms, and a Gamma-only cell)."""
    from dataclasses import replace
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=7) if cell else ki.small_binary().systems[0]
    nu, eig = ph.phonons(s, mesh)
    pair = np.any(s.fc3_idx[:, 2:5] != 0, axis=1) | np.any(s.fc3_idx[:, 6:9] != 0, axis=1)
    b = int(np.argmax(np.where(pair, np.abs(s.fc3).max(axis=(1, 2, 3)), 0.0)))
    fc3 = s.fc3.copy()
    fc3[b] *= 2.0
    added = replace(s, fc3=fc3)
    twice = replace(s, fc3=np.concatenate([s.fc3, s.fc3[b:b + 1]]),
                    fc3_idx=np.concatenate([s.fc3_idx, s.fc3_idx[b:b + 1]]))
    ref, _ = kk.kald_linewidths(ctx, [added], mesh, nu.ravel(), eig.ravel(),
                                kk.Options(temperature_K=300.0, sigma_thz=0.1, precision="fp64", symmetry="none"))
    got, _ = kk.kald_linewidths(ctx, [twice], mesh, nu.ravel(), eig.ravel(),
                                kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=precision))
    assert _rel(got, ref) < (1e-10 if precision == "fp64" else 1e-5)


def _two_parts(cell, ratio, mix):
    """Two copies of a cell in one, the second with Phi2 0.81 and Phi3 `ratio` times the
    first's and no force between them (nor a mode of one in a degenerate set with one of
    the other, whose linewidths would be averaged); with `mix`, pairs of modes of the two (of nearly
    one frequency) rotated into each other and given their mean frequency."""
    from dataclasses import replace
    a = ki.fcc_supercell_system(cell, seed=5)
    n = a.n_atoms
    i2, i3 = a.fc2_idx.copy(), a.fc3_idx.copy()
    i2[:, :2] += n
    i3[:, [0, 1, 5]] += n
    s = replace(a, masses=np.tile(a.masses, 2), positions=np.concatenate([a.positions, a.positions + 1.3]),
                fc2_idx=np.concatenate([a.fc2_idx, i2]), fc2=np.concatenate([a.fc2, 0.81 * a.fc2]),
                fc3_idx=np.concatenate([a.fc3_idx, i3]), fc3=np.concatenate([a.fc3, ratio * a.fc3]))
    nu, eig = ph.phonons(a, (1, 1, 1))
    nb = 3 * n
    nu2 = np.concatenate([nu[0], 0.9 * nu[0]])
    E = np.zeros((2 * nb, 2 * nb))
    E[:nb, :nb] = E[nb:, nb:] = eig[0].real
    part = np.repeat([0, 1], nb)
    if mix:
        # every fourth mode of the first part from the 10th with the mode of the second nearest to it
        left = set(range(nb + 10, 2 * nb))
        for m in range(10, nb, 4):
            o = min(left, key=lambda x: abs(nu2[x] - nu2[m]))
            left.remove(o)
            E[m], E[o] = (E[m] + E[o]) / np.sqrt(2), (E[m] - E[o]) / np.sqrt(2)
            nu2[m] = nu2[o] = 0.5 * (nu2[m] + nu2[o])
            nu2[o] += 1e-3                           # (not a degenerate set)
            part[[m, o]] = 2
    order = np.argsort(nu2, kind="stable")
    other = (part[order][1:] != part[order][:-1]) & (nu2[order][1:] > 0.01)
    assert np.diff(nu2[order])[other].min() > 1e-5
    return s, nu2[order][None], E[order].astype(complex)[None], part[order]


@pytest.mark.parametrize("symmetry", ["all", "inversion"])
@pytest.mark.parametrize("mix", [False, True])
@pytest.mark.parametrize("log_ratio", [0, 12, 20, 24])
def test_gamma_only_split_of_unlike_parts(k, log_ratio, mix, symmetry):
    """A part whose Phi3 is up to 2^24 times weaker than the rest of the cell keeps the
    linewidths of its modes (gamma 2^48 times smaller: each part is compared with its own
    largest) to the 1e-5 of the mode, as do modes that extend over both parts; each triple
    of modes projected once and three times."""
    kk, ctx = k
    s, nu, eig, part = _two_parts((3, 3, 1), 2.0 ** -log_ratio, mix)
    out = {}
    for prec in ("fp64", "bf16split"):
        opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=prec, symmetry=symmetry)
        out[prec] = kk.kald_linewidths(ctx, [s], (1, 1, 1), nu.ravel(), eig.ravel(), opt)
    assert abs(out["fp64"][1][1] - out["bf16split"][1][1]) <= 1e-5 * out["fp64"][1][1]
    ref, got = (np.asarray(out[p][0]).ravel() for p in ("fp64", "bf16split"))
    for x in set(part):
        assert _rel(got[part == x], ref[part == x]) < 1e-5


def test_orbit_sums_of_a_dense_mesh(k):
    """Three atoms on 20^3: 5.3 million orbits whose positions' sums would take 1.15 GB.
    They are projected in several launches, so that the context holds less than a GB for
    them all with everything else (256 MB of sums, 0.4 GB of tables and orbits), and the
    linewidths are those of single q-points, which use time reversal only."""
    torch = pytest.importorskip("torch")
    from kald_inputs.configs import A_FCC
    from kald_inputs.lattice import fcc_primitive
    from kald_inputs.lj import lj_system
    kk, _ = k
    lat = fcc_primitive(A_FCC)[0]
    s = lj_system(lat * np.array([3, 1, 1])[:, None], np.arange(3)[:, None] * lat[:1], [39.948, 60.0, 39.948])
    mesh = (20, 20, 20)
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision="fp64")
    with kk.Context(0) as ctx:
        nu, eig, _ = kk.kald_phonons(ctx, s, mesh, want_vel=False)
        qs = [1, 777, 4210, 7999]
        ref, _ = kk.kald_linewidths_qlist(ctx, s, mesh, nu.ravel(), eig.ravel(), opt, qs)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with kk.Context(0) as ctx:
        g, _ = kk.kald_linewidths(ctx, s, mesh, nu.ravel(), eig.ravel(), opt)
        held = free - torch.cuda.mem_get_info()[0]
    assert held < 1 << 30
    g = np.asarray(g).reshape(8000, 9)[qs]
    assert _rel(g, np.asarray(ref).reshape(g.shape)) < 1e-10


@pytest.mark.parametrize("cell", [(1, 1, 1), (3, 3, 1), (11, 1, 1), (5, 3, 3)])
def test_generalised_velocities_workspace(k, cell):
    """12, 108, 132 and 540 modes (whole tiles and small remainders): the smallest
    workspace of the calls is no more than that of the product in FP64 matrices would be
    (E, three B and three W, the blocks as given and mass-scaled)."""
    import re
    torch = pytest.importorskip("torch")
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=5)
    nb, n2 = s.n_branches, len(s.fc2)
    up = lambda *b: sum(-(-x // 256) * 256 for x in b)
    fc2 = up(4 * (s.n_atoms + 1), 4 * n2, 72 * n2, 8 * n2, 8 * s.n_atoms, 72 * n2, 24 * n2)
    mats = up(8 * nb * nb, 24 * nb * nb, 24 * nb * nb)
    n_partial = min(nb, 4 * torch.cuda.get_device_properties(0).multi_processor_count)
    nu, eig = ph.phonons(s, (1, 1, 1))
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (nu.ravel(), eig.ravel(), np.full(nb, 0.1))]
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1)
    for call, rest in ((lambda: kk.kald_diffusivity(ctx, [s], *dev, opt, torch.zeros(nb, dtype=torch.float64).cuda()),
                        up(8 * nb) * 2),
                       (lambda: kk.kald_kappa_qhgk(ctx, [s], *dev, opt), up(8 * (9 * n_partial + nb), 72))):
        ctx.set_workspace_limit(1)
        try:
            with pytest.raises(kk.KaldError) as e:
                call()
        finally:
            ctx.set_workspace_limit(0)
        assert int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)) <= fc2 + mats + rest


@pytest.mark.parametrize("symmetry", ["all", "none"])
@pytest.mark.parametrize("cell,mesh,precision", [(None, (2, 1, 1), "fp32"), ((1, 1, 1), (2, 1, 1), "fp32"),
                                                 ((3, 1, 1), (1, 1, 1), "fp64"), ((2, 2, 2), (2, 1, 1), "bf16split")])
def test_window_edges_at_high_frequencies(k, cell, mesh, precision, symmetry):
    """Two frequencies f1 of 200 to 300 THz and f2, |2 f1 - f2| inside the window of a
    0.004 THz delta by 1e-5 of its width, where a rounding of FP32 sums of the
    frequencies is 1e-4 rad/ps: the coarse tests of whole tiles drop none of the triplets,
    (f1, f1, f2) and (f2, f1, f1), that the exact test takes."""
    kk, ctx = k
    s = ki.fcc_supercell_system(cell, seed=7) if cell else ki.small_binary().systems[0]
    _, eig = ph.phonons(s, mesh)
    nb, nq = s.n_branches, int(np.prod(mesh))
    n1 = nb // 2
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.004, precision=precision, symmetry=symmetry)
    for x in np.random.default_rng(nb).uniform(200.0, 300.0, 24):
        for sign in (1.0, -1.0):
            nu = np.full((nq, nb), x)
            nu[:, n1:] = 2.0 * x + sign * 0.012 * (1.0 - 1e-5)
            _, count = kk.kald_linewidths(ctx, s, mesh, nu, eig, opt)
            assert count[1] == nq * nq * 2 * n1 * n1 * (nb - n1)


@pytest.mark.parametrize("top,sigma,change", [(50.0, 0.05, 3e-13), (20.0, 0.01, 3e-13), (50.0, 0.05, 4e-15), (2.0, 20.0, 3e-13)])
def test_phase_space_mirrored_within_the_window(k, top, sigma, change):
    """Spectra much wider than the delta, and a delta wider than the spectrum: frequencies
    of -q that differ from those of q by `change` of the largest change no sum by more
    than 1e-10, whether those of q are taken for both or not (the smallest workspace sums
    every q-point by itself)."""
    import re
    kk, ctx = k
    mesh, nb = (4, 3, 2), 6
    s = ki.small_binary(mesh=mesh).systems[0]
    nq = int(np.prod(mesh))
    rng = np.random.default_rng(5)
    nu = np.sort(rng.uniform(0.02, top, (nq, nb)), axis=1)
    nu[:, 0], nu[:, -1] = 0.011, top
    neg = np.array([np.ravel_multi_index(tuple((-np.array(np.unravel_index(q, mesh))) % mesh), mesh) for q in range(nq)])
    # triplets at every place of the window: the middle modes of every q near half of the top
    nu[:, 2:5] = 0.5 * top + sigma * rng.uniform(-1.0, 1.0, (nq, 3))
    nu = np.where((neg < np.arange(nq))[:, None], nu[neg] + change * top * rng.choice([-1.0, 1.0], (nq, nb)), nu)
    opt = kk.Options(temperature_K=300.0, sigma_thz=sigma, precision="fp64")
    g = kk.kald_phase_space(ctx, s, mesh, nu, opt)
    ctx.set_workspace_limit(1)
    try:
        with pytest.raises(kk.KaldError) as e:
            kk.kald_phase_space(ctx, s, mesh, nu, opt)
        ctx.set_workspace_limit(int(re.search(r"needs (\d+) bytes", str(e.value)).group(1)))
        ref = kk.kald_phase_space(ctx, s, mesh, nu, opt)
    finally:
        ctx.set_workspace_limit(0)
    assert np.max(np.abs(g - ref)) <= 1e-10 * np.max(np.abs(ref))


def test_phonons_of_more_systems_than_are_planned_at_once(k):
    """70 Gamma-only systems, all different, large ones among small ones at both ends of
    the 64 that are planned together: the phonons of each alone, bit for bit."""
    from dataclasses import replace
    kk, ctx = k
    base, big = ki.fcc_supercell_system((1, 1, 1), seed=3), ki.fcc_supercell_system((3, 3, 1), seed=9)
    systems = [replace(big if x in (0, 31, 64, 69) else base, masses=(big if x in (0, 31, 64, 69) else base).masses + 0.01 * x)
               for x in range(70)]
    nu, eig = kk.kald_phonons_batch(ctx, systems)
    o = e = 0
    for s in systems:
        nb = s.n_branches
        nu1, eig1, _ = kk.kald_phonons(ctx, s, (1, 1, 1), want_vel=False)
        np.testing.assert_array_equal(np.asarray(nu).ravel()[o:o + nb], nu1.ravel())
        np.testing.assert_array_equal(np.asarray(eig).ravel()[e:e + nb * nb], eig1.ravel())
        o += nb
        e += nb * nb
    bad = replace(base, masses=-base.masses)
    with pytest.raises(kk.KaldError, match="masses"):
        kk.kald_phonons_batch(ctx, systems[:66] + [bad])


def test_symmetry_of_a_weak_part(k):
    """A part of a cell whose force constants are 2^-30 (Phi3) and 2^-24 (Phi2) of the
    other's and lack the symmetry by 1e-4 and 1e-5 of themselves, less than 1e-12 of the
    largest: neither is taken as symmetric, and the part's linewidths and generalised
    velocities are those of its own force constants (1e-10 of the part's largest)."""
    from dataclasses import replace
    from oracle import conductivity as co
    kk, ctx = k
    rng = np.random.default_rng(3)
    s, _, _, _ = _two_parts((1, 1, 1), 2.0 ** -30, False)
    n = s.n_atoms // 2
    weak = s.fc3_idx[:, 0] >= n
    s = replace(s, fc3=np.where(weak[:, None, None, None], s.fc3 * (1.0 + 1e-4 * rng.standard_normal(s.fc3.shape)), s.fc3))
    mesh = (2, 2, 1)
    nu, eig = ph.phonons(s, mesh)
    of_weak = (np.abs(eig[:, :, 3 * n:]) ** 2).sum(-1).ravel() > 0.5
    g = [np.asarray(kk.kald_linewidths(ctx, s, mesh, nu, eig, kk.Options(temperature_K=300.0, sigma_thz=0.1, precision="fp64",
                                                                         symmetry=sym))[0]).ravel()
         for sym in ("all", "none")]
    for part in (of_weak, ~of_weak):
        assert _rel(g[0][part], g[1][part]) < 1e-10

    s, _, _, _ = _two_parts((2, 2, 1), 1.0, False)
    n = s.n_atoms // 2
    weak = (s.fc2_idx[:, 0] >= n)[:, None, None]
    s = replace(s, fc2=np.where(weak, 2.0 ** -24 * s.fc2 * (1.0 + 1e-5 * rng.standard_normal(s.fc2.shape)), s.fc2))
    # any orthonormal modes, each on one part
    E = np.zeros((6 * n, 6 * n))
    E[:3 * n, :3 * n], E[3 * n:, 3 * n:] = (np.linalg.qr(rng.standard_normal((3 * n, 3 * n)))[0] for _ in range(2))
    eig = E.astype(complex)[None]
    nu = np.sort(rng.uniform(0.1, 2.0, (1, 6 * n)))
    W_o = co.generalized_velocity(s, nu, eig)[:, 3 * n:, 3 * n:]
    _, W = kk.kald_kappa_qhgk(ctx, [s], nu.ravel(), eig.ravel(), np.full(6 * n, 0.1),
                              kk.Options(temperature_K=300.0, sigma_thz=0.1), want_vgen=True)
    np.testing.assert_allclose(W[:, 3 * n:, 3 * n:], W_o, rtol=0, atol=1e-10 * np.abs(W_o).max())


@pytest.mark.parametrize("phase_sum", ["0", "1"])
@pytest.mark.parametrize("log_ratio", [20, 24])
def test_crystal_split_of_unlike_parts(k, log_ratio, phase_sum, monkeypatch):
    """72 branches, half of them on a part whose Phi3 is 2^20 or 2^24 times weaker, with
    the phase sum on CUDA cores and on tensor cores: a power of two in a part's Phi3 is
    exact in every operand, so the part's linewidths are those of the same cell with
    parts of one strength times its square, to the rounding of FP32 sums."""
    kk, ctx = k
    monkeypatch.setenv("KALD_TCX_Y", phase_sum)
    mesh = (3, 1, 1)
    opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision="bf16split")
    alike, unlike = (_two_parts((3, 1, 1), r, False)[0] for r in (1.0, 2.0 ** -log_ratio))
    nu, eig = ph.phonons(alike, mesh)
    weak = (np.abs(eig[:, :, 36:]) ** 2).sum(-1).ravel() > 0.5
    ref, got = (np.asarray(kk.kald_linewidths(ctx, s, mesh, nu, eig, opt)[0]).ravel() for s in (alike, unlike))
    assert _rel(got[weak] * 4.0 ** log_ratio, ref[weak]) < 1e-6
    assert _rel(got[~weak], ref[~weak]) < 1e-6


@pytest.mark.parametrize("cell,extra", [((3, 3, 1), 12000), ((9, 1, 1), 40000), ((13, 1, 1), 2500)])
def test_gamma_only_y_build_of_dense_cells(k, cell, extra):
    """Atom pairs of 1 to some 45 blocks each, all pairs of the cell in use: outputs of a
    lane, of three lanes of a warp and of all warps of a CTA in one set of rows (108 and
    156 modes; a Phi3 without symmetry)."""
    kk, ctx = k
    s = ki.random_fc3_system(ki.fcc_supercell_system(cell, seed=5), extra, seed=3)
    nu, eig = ph.phonons(s, (1, 1, 1))
    out = {}
    for prec in ("fp64", "bf16split"):
        opt = kk.Options(temperature_K=300.0, sigma_thz=0.1, precision=prec)
        out[prec] = kk.kald_linewidths(ctx, [s], (1, 1, 1), nu.ravel(), eig.ravel(), opt)
    assert abs(out["fp64"][1][1] - out["bf16split"][1][1]) <= 1e-5 * out["fp64"][1][1]
    assert _rel(out["bf16split"][0], out["fp64"][0]) < 1e-5
