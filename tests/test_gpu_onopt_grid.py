"""The occupation optimiser spreads the subspaces over a grid: shapes at the edges of that
mapping (one subspace, one weak orbital per subspace, the largest N_g, more subspaces than
SMs would take, row sums over chunks with a remainder) against the oracle's E(gamma) and
dE/dgamma.  Tolerance: both sum the same terms in FP64 in different orders, so E differs by
at most about N_Omega^2 roundings of its largest partial sum: 1e-12 of the sum of the
terms' magnitudes, which 1e-11 |E| + 1e-11 bounds here; the gradient likewise of its scale."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import integrals as I, onopt, ri  # noqa: E402
from synthetic import (draw_gamma, make_system, orthonormal_orbitals, pairing_columns,  # noqa: E402
                       random_orthogonal, without_basis_functions)


@pytest.mark.parametrize("n_c,n_strong,n_weak,naux", [(3, 1, 1, 40), (3, 1, 16, 40), (3, 4, 16, 40), (3, 13, 4, 60),
                                                      (5, 20, 5, 60), (14, 160, 1, 60)])
def test_energy_and_gradient_on_every_grid_shape(n_c, n_strong, n_weak, naux):
    from paper_2012_15662_gb300 import binding as bd
    full = make_system("ring", n_c=n_c, seed=5, n_weak_per=1)
    s = dataclasses.replace(without_basis_functions(full, 0, full.naux - naux), n_strong=n_strong, n_weak_per=n_weak)
    assert s.n_omega <= s.nbf
    rng = np.random.default_rng(31 + n_strong)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(s.nbf, rng))
    gamma = draw_gamma(n_strong, n_weak, rng, 0.2, 1.3)
    sub, rank = pairing_columns(n_strong, n_weak)
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    eng.transform(C, bd.DONOF_RI_FULL)
    J, K = eng.jk_mo()
    g, E, grad, it, reason = eng.optimize_occupations(gamma, max_iter=0)
    again = eng.optimize_occupations(gamma, max_iter=3)
    assert again[3] <= 3 and again[1] <= E
    eng.close()
    m = s.n_omega
    Hd = np.einsum("mp,mn,np->p", C[:, :m], I.core_hamiltonian(s), C[:, :m])
    E_ref, g_ref = onopt.energy_and_gradient(gamma, n_strong, n_weak, sub, rank, Hd, J, K, I.nuclear_repulsion(s))
    assert np.array_equal(g, gamma) and it == 0
    assert abs(E - E_ref) <= 1e-11 * abs(E_ref) + 1e-11
    assert np.abs(grad - g_ref).max() <= 1e-10 * np.abs(g_ref).max()
