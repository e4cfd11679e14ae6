"""The error of FP64 products from digit planes, against the engine's own operands in extended
precision (so that no conditioning enters): at the edges of the K chunks (128 elements, two
accumulator sets in turn) and K blocks (32), and with operands whose rows are graded against one
another, where the small elements of one meet the large ones of the other.

Bound of an output sum_k A_k B_k, with a = max|A|, b = max|B|.  An operand row becomes integers of 62
bits under 2^e, 2^e <= 4 a, rounded to nearest: an element is off by 2^(e - 63) <= 2^-61 a, the output by
2^-61 (a sum|B| + b sum|A|).  The digit pairs left out (t + u >= 8; five of weight 2^-72, each at most
2^16 in units of 2^(ea + eb - 16) <= 2^-12 a b) give K 5 2^-72 2^16 2^-12 a b < 2^-65 K a b.  One rounding
of the result: 2^-53 of it (by integers, good to 2^-11 of that).  Integers up to 2^24 per chunk are exact
in the accumulators; random digits stay below."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import integrals as I  # noqa: E402
from synthetic import make_system, orthonormal_orbitals, random_orthogonal, without_basis_functions  # noqa: E402


def _check(got, A, B):
    """got[i] against sum_k A[i, k] B[i, k]."""
    q = np.longdouble
    ref = (A.astype(q) * B.astype(q)).sum(1)
    a, b = np.abs(A).max(1), np.abs(B).max(1)
    bound = (2.0**-61 * (a * np.abs(B).sum(1) + b * np.abs(A).sum(1)) + 2.0**-65 * A.shape[1] * a * b
             + (1 + 2.0**-9) * 2.0**-53 * np.abs(ref).astype(float))
    err = np.abs(got.astype(q) - ref).astype(float)
    assert (err <= bound).all(), (err / np.maximum(bound, 1e-300)).max()


def _system(n_c, nbf, naux, weak):
    full = make_system("ring", n_c=n_c, seed=5, n_weak_per=weak)
    return without_basis_functions(full, full.nbf - nbf, full.naux - naux)


@pytest.mark.parametrize("n_c,nbf,naux", [(5, 120, 256), (5, 120, 257), (5, 119, 288), (5, 120, 289), (6, 144, 320),
                                          (7, 161, 511), (7, 160, 513)])
def test_sums_over_the_auxiliary_index(n_c, nbf, naux):
    from paper_2012_15662_gb300 import binding as bd
    s = _system(n_c, nbf, naux, 4)
    rng = np.random.default_rng(naux)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(nbf, rng))
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    eng.transform(C, bd.DONOF_RI_FULL)
    d, bh, B = (eng.fetch(w) for w in (bd.DONOF_RI_FETCH_DIAG, bd.DONOF_RI_FETCH_BHALF, bd.DONOF_RI_FETCH_B))
    J, _ = eng.jk_mo()
    Jao, Kao = eng.jk_ao()
    eng.close()
    p, q = rng.integers(0, s.n_omega, (2, 500))
    mu, nu = rng.integers(0, nbf, (2, 500))
    _check(J[p, q], d[:, p].T, d[:, q].T)
    _check(Jao[q, mu, nu], d[:, q].T, B[:, mu, nu].T)
    _check(Kao[q, mu, nu], bh[:, q, mu].T, bh[:, q, nu].T)


@pytest.mark.parametrize("n_c,nbf", [(4, 96), (5, 97), (5, 120), (6, 127), (6, 129), (8, 192), (8, 191)])
@pytest.mark.parametrize("orbitals", ["spread", "local", "graded"])
def test_half_transform(n_c, nbf, orbitals):
    """b_half of orthonormal orbitals spread over the ring, of the ones nearest to the basis
    functions (S^-1/2), and of columns that fall by 2^40 from one function to the last."""
    from paper_2012_15662_gb300 import binding as bd
    s = _system(n_c, nbf, 260, 2)
    rng = np.random.default_rng(nbf)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(nbf, rng) if orbitals == "spread" else np.eye(nbf))
    if orbitals == "graded":
        order = np.stack([rng.permutation(nbf) for _ in range(nbf)], 1)
        C = rng.standard_normal((nbf, nbf)) * 2.0 ** (-40.0 * order / nbf)
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    eng.transform(C, bd.DONOF_RI_HALF)
    bh, B = eng.fetch(bd.DONOF_RI_FETCH_BHALF), eng.fetch(bd.DONOF_RI_FETCH_B)
    eng.close()
    P, p, nu = rng.integers(0, s.naux, 800), rng.integers(0, s.n_omega, 800), rng.integers(0, nbf, 800)
    _check(bh[P, p, nu], C[:, p].T, B[P, nu, :])
