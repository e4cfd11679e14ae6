"""FP64 products from digit planes on the tensor cores, through the calls that use them, at
the edges of their tiles (128 x 32 outputs, K blocks of 32, K chunks of 256) and of their
rules (96 functions; 256 auxiliary functions for the fit).

Tolerances.  Rotation: C expm(kappa) against scipy's expm.  About 13 products, each off by a
few 2^-53 of |A||B|; with ||kappa|| of order 1 and orthonormal rows that is below
13 * n * 2^-53 per element (3e-13 at 200), plus the re-orthonormalisation's own rounding: 1e-11
of the largest orbital coefficient.  Fit: residual L X - R of the solved B against the
three-centre integrals, elementwise below 8 n 2^-53 |L||X| (substitution itself gives n 2^-53)."""
import numpy as np
import pytest
from scipy.linalg import expm

pytestmark = pytest.mark.gpu

from oracle import integrals as I  # noqa: E402
from synthetic import make_system, orthonormal_orbitals, random_orthogonal, without_basis_functions  # noqa: E402


@pytest.mark.parametrize("nbf,norm", [(95, 0.3), (96, 1e-3), (97, 3.0), (128, 0.5), (129, 20.0), (161, 1.0), (192, 0.0)])
def test_rotation_at_tile_edges(nbf, norm):
    from paper_2012_15662_gb300 import binding as bd
    n_c = (nbf + 23) // 24
    full = make_system("ring", n_c=n_c, seed=7, n_weak_per=1)
    s = without_basis_functions(full, full.nbf - nbf, full.naux - 40)
    rng = np.random.default_rng(nbf)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(nbf, rng))
    k = rng.standard_normal((nbf, nbf))
    k = k - k.T
    k *= norm / np.linalg.norm(k, 2)
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    eng.transform(C, bd.DONOF_RI_HALF)
    out = np.empty(nbf * nbf)
    bd.donof_ri_apply_rotation(eng.ctx, k, out)
    C1 = out.reshape(nbf, nbf).T
    eng.close()
    ref = C @ expm(k)
    assert np.abs(C1 - ref).max() <= 1e-11 * np.abs(C).max()


@pytest.mark.parametrize("n_c,drop_bf,drop_aux", [(3, 0, 0), (4, 33, 0), (4, 32, 80), (4, 31, 79), (4, 0, 0), (5, 0, 36),
                                                  (5, 7, 35), (6, 1, 0)])
def test_fit_solves_the_triangular_system(n_c, drop_bf, drop_aux):
    from paper_2012_15662_gb300 import binding as bd
    s = without_basis_functions(make_system("ring", n_c=n_c, seed=3, n_weak_per=1), drop_bf, drop_aux)
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    X = eng.fetch(bd.DONOF_RI_FETCH_B).reshape(s.naux, s.nbf, s.nbf)
    L = np.tril(eng.fetch(bd.DONOF_RI_FETCH_METRIC).reshape(s.naux, s.naux))
    eng.close()
    # every column stands alone: a sample of them, the corners among them, in extended precision
    cols = np.unique(np.r_[0, s.nbf - 1, s.nbf * s.nbf - 1, np.random.default_rng(1).integers(0, s.nbf * s.nbf, 800)])
    R = I.eri3(s).reshape(s.naux, -1)[:, cols]
    x = X.reshape(s.naux, -1)[:, cols]
    assert np.abs(X - X.transpose(0, 2, 1)).max() <= 1e-11 * np.abs(X).max()
    # the integrals themselves are good to a few roundings of their largest factor
    res = np.abs(L.astype(np.longdouble) @ x.astype(np.longdouble) - R).astype(float)
    bound = 8 * s.naux * 2.0**-53 * (np.abs(L) @ np.abs(x)) + 1e-14 * np.abs(R).max()
    assert (res <= bound).all(), (res / bound).max()


@pytest.mark.parametrize("n_c,drop_bf", [(4, 0), (4, 1), (5, 0), (6, 15)])
def test_working_basis_gives_the_same_coulomb_matrix(n_c, drop_bf):
    """J_pq of the digit engine (working basis from the products) against FP64's: the engine's
    own quantisation is 2^-31 of each row's largest element, 1e-7 of the largest J."""
    from paper_2012_15662_gb300 import binding as bd
    s = without_basis_functions(make_system("ring", n_c=n_c, seed=9, n_weak_per=2), drop_bf, 0)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(s.nbf, np.random.default_rng(2)))
    out = []
    for prec in (bd.DONOF_RI_FP64, bd.DONOF_RI_SLICE4):
        eng = bd.Engine(s, prec)
        eng.transform(C, bd.DONOF_RI_FULL)
        out.append(eng.jk_mo())
        eng.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-7 * np.abs(a).max()


@pytest.mark.parametrize("n_c,weak,drop_bf,drop_aux", [(4, 4, 0, 80), (4, 4, 0, 81), (4, 1, 1, 0), (5, 3, 7, 0)])
def test_fp64_iteration_on_both_sides_of_the_rule(n_c, weak, drop_bf, drop_aux):
    """The FP64 precision's products come from digits at 256 auxiliary functions and from FP64
    FMAs at 255: J, K, E and lambda against the oracle.  Both are FP64-accurate; B carries the
    metric's condition (about 1e7, 1e-9 of its elements as in the other FP64 tests)."""
    from oracle import pnof7, ri
    from paper_2012_15662_gb300 import binding as bd
    from synthetic import draw_gamma, pairing_columns
    s = without_basis_functions(make_system("ring", n_c=n_c, seed=4, n_weak_per=weak), drop_bf, drop_aux)
    rng = np.random.default_rng(8)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(s.nbf, rng))
    gamma = draw_gamma(s.n_strong, s.n_weak_per, rng)
    m = s.n_omega
    B, _, _ = ri.setup(s)
    rows = ri.all_rows(B, C, m)
    sub, rank = pairing_columns(s.n_strong, s.n_weak_per)
    n = pnof7.occupations(gamma, s.n_strong, s.n_weak_per, sub, rank)
    A, Bc = pnof7.coupling(n, sub, rank)
    H = I.core_hamiltonian(s)
    lam = pnof7.lagrangian(C, H, rows["Jao"], rows["Kao"], n, A, Bc)
    E = pnof7.energy(n, np.einsum("mp,mn,np->p", C[:, :m], H, C[:, :m]), rows["J"], rows["K"], A, Bc,
                     I.nuclear_repulsion(s))
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    eng.transform(C, bd.DONOF_RI_FULL)
    J, K = eng.jk_mo()
    Jao, Kao = eng.jk_ao()
    E1, lam1 = eng.energy_lagrangian(gamma)
    eng.close()
    for a, b in ((J, rows["J"]), (K, rows["K"]), (Jao, rows["Jao"]), (Kao, rows["Kao"])):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
    assert abs(E1 - E) <= 1e-9 * abs(E)
    assert np.abs(lam1 - lam).max() <= 1e-9 * np.abs(lam).max()
