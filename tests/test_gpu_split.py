"""The digits of J^(q) and K^(q) taken in one pass (a matrix's triangle in shared memory, up to
240 functions) and in two (above): sizes around the rules on threads and shared memory, odd
ones (the middle row stands alone on its line) and remainders of the groups of four, through
the Lagrangian they feed, against the FP64 precision.  The digit engine quantises each row at
2^-31 of its largest element, so E and lambda agree to 1e-7 of their largest entry (a wrong
or missing element shows at 1e-2)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import integrals as I  # noqa: E402
from synthetic import draw_gamma, make_system, orthonormal_orbitals, random_orthogonal, without_basis_functions  # noqa: E402


@pytest.mark.parametrize("n_c,nbf", [(3, 41), (3, 47), (3, 48), (3, 49), (5, 113), (7, 165), (7, 166), (7, 167), (10, 239),
                                     (10, 240), (11, 241)])
def test_lagrangian_from_the_digits_of_each_size(n_c, nbf):
    from paper_2012_15662_gb300 import binding as bd
    full = make_system("ring", n_c=n_c, seed=6, n_weak_per=1)
    s = without_basis_functions(full, full.nbf - nbf, full.naux - 70)
    rng = np.random.default_rng(nbf)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(nbf, rng))
    gamma = draw_gamma(s.n_strong, s.n_weak_per, rng)
    out = []
    for prec in (bd.DONOF_RI_FP64, bd.DONOF_RI_SLICE4):
        eng = bd.Engine(s, prec)
        eng.transform(C, bd.DONOF_RI_HALF)
        eng.jk_ao()
        out.append(eng.energy_lagrangian(gamma))
        eng.close()
    (E0, l0), (E1, l1) = out
    assert abs(E1 - E0) <= 1e-7 * abs(E0)
    assert np.abs(l1 - l0).max() <= 1e-7 * np.abs(l0).max()
