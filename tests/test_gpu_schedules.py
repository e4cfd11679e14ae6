"""Every pipeline depth and both unit lists of the digit-plane GEMMs, at an odd number of column
tiles (N_Omega 120: three) and ragged rows.

Digits, J^(q), K^(q) and J (exact integer sums) do not depend on the schedule.  K_pq, F^(p) C_p and so
lambda and E are double-float sums in the order of the units: a double-float addition is off by at most
2^-44 of its result, so two orders of n terms t differ by at most 2 n 2^-44 sum|t|.  K_pq sums naux
squares, for which sum|t| is K_pq itself.  F^(p) C_p sums 2 N_Omega + 1 vectors, n_p H C_p, A_pq J^(q) C_p
and B_pq K^(q) C_p; in the working basis, where C is orthogonal, the norm of a vector is that of its
products with all orbitals, and the difference of lambda's column p is at most 2 (2 N_Omega + 1) 2^-44
times the sum of those norms, and nbf 2^-44 twice more for the products with C themselves.  E takes the
sum of these over p."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import integrals as I, pnof7  # noqa: E402
from synthetic import (draw_gamma, make_system, orthonormal_orbitals, pairing_columns, random_orthogonal,  # noqa: E402
                       without_basis_functions)

HALF, FULL, JMO, JAO, KAO, FOCK = range(6)


def test_results_do_not_depend_on_the_schedule():
    from paper_2012_15662_gb300 import binding as bd
    full = make_system("ring", n_c=6, seed=8, n_weak_per=4)
    s = without_basis_functions(full, 7, 21)
    assert (s.nbf, s.n_omega) == (137, 120)
    rng = np.random.default_rng(8)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(s.nbf, rng))
    gamma = draw_gamma(s.n_strong, s.n_weak_per, rng)
    eng = bd.Engine(s, bd.DONOF_RI_SLICE4)

    def run():
        eng.transform(C, bd.DONOF_RI_FULL)
        J, K = eng.jk_mo()
        bh = eng.fetch(bd.DONOF_RI_FETCH_BHALF)
        Jao, Kao = eng.jk_ao()
        E, lam = eng.energy_lagrangian(gamma)
        return J, bh, Jao, Kao, K, lam, E

    ref = run()
    nb, m = s.nbf, s.n_omega
    sub, rank = pairing_columns(s.n_strong, s.n_weak_per)
    n = pnof7.occupations(gamma, s.n_strong, s.n_weak_per, sub, rank)
    A, B = pnof7.coupling(n, sub, rank)
    norm = {k: np.linalg.norm(np.einsum("mr,qmn,np->qrp", C, X, C[:, :m], optimize=True), axis=1)
            for k, X in (("J", ref[2]), ("K", ref[3]), ("H", I.core_hamiltonian(s)[None]))}
    size = n * norm["H"][0] + (np.abs(A).T * norm["J"]).sum(0) + (np.abs(B).T * norm["K"]).sum(0)
    bound = (2 * (2 * m + 1) + 2 * nb) * 2.0**-44 * size
    for stages in (2, 3, 4):
        for opt in (1, 2):
            for kind in range(6):
                option = {HALF: 1, JAO: opt - 1, KAO: opt - 1}.get(kind, opt)
                bd.donof_ri_set_schedule(eng.ctx, kind, stages, option)
            out = run()
            for a, b in zip(out[:4], ref[:4]):
                np.testing.assert_array_equal(a, b)
            assert (np.abs(out[4] - ref[4]) <= 2 * s.naux * 2.0**-44 * ref[4]).all()
            assert (np.abs(out[5] - ref[5])[:, :m].max(0) <= bound).all()
            assert abs(out[6] - ref[6]) <= bound.sum()
    eng.close()
