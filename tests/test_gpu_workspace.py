"""Which arithmetic the FP64 products take is a matter of sizes, not of the device memory that
happens to be free: with room for half, a tenth and hardly any of the workspace a context or a
rotation would like, the results are the same to the bit."""
import gc

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import integrals as I  # noqa: E402
from synthetic import draw_gamma, make_system, orthonormal_orbitals, random_orthogonal, without_basis_functions  # noqa: E402

MB = 1 << 20


class _LittleMemory:
    """Leaves `free` bytes of device memory to the code inside."""

    def __init__(self, free):
        self.free = free

    def __enter__(self):
        import torch
        torch.cuda.empty_cache()
        have = torch.cuda.mem_get_info()[0]
        self.hold = torch.empty(max(0, have - self.free) // MB * MB, dtype=torch.uint8, device="cuda")
        return self

    def __exit__(self, *_):
        import torch
        del self.hold
        gc.collect()
        torch.cuda.empty_cache()


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_fp64_context_with_little_memory():
    from paper_2012_15662_gb300 import binding as bd
    s = make_system("ring", n_c=6, seed=4, n_weak_per=4)  # 144 / 504 / 120: digits of b_half's operands 163 MB
    rng = np.random.default_rng(3)
    C = orthonormal_orbitals(I.overlap(s), random_orthogonal(s.nbf, rng))
    gamma = draw_gamma(s.n_strong, s.n_weak_per, rng)

    def run(eng):
        eng.transform(C, bd.DONOF_RI_FULL)
        J, K = eng.jk_mo()
        eng.jk_ao(want=False)
        E, lam = eng.energy_lagrangian(gamma)
        return J, K, E, lam

    bd.Engine(s, bd.DONOF_RI_FP64).close()  # whatever the library allocates once
    before = _free()
    eng = bd.Engine(s, bd.DONOF_RI_FP64)
    used = before - _free()
    ref = run(eng)
    eng.close()
    digits = s.naux * s.nbf * 14 * (s.nbf + 16)
    for share in (0.6, 0.15, 0.06):
        with _LittleMemory(used - int((1 - share) * digits)):
            eng = bd.Engine(s, bd.DONOF_RI_FP64)
            out = run(eng)
            eng.close()
        for a, b in zip(out, ref):
            np.testing.assert_array_equal(a, b)


def test_rotation_with_little_memory():
    """720 functions: scratch of 24 MB, digits of both operands 14 MB, of one with 128 rows of the
    other 8.2 MB."""
    from paper_2012_15662_gb300 import binding as bd
    nbf = 720
    full = make_system("ring", n_c=20, seed=4, n_weak_per=1)
    s = without_basis_functions(full, 0, full.naux - 32)
    rng = np.random.default_rng(5)
    C = random_orthogonal(nbf, rng)
    k = rng.standard_normal((nbf, nbf))
    k = 0.01 * (k - k.T)
    out = [np.empty(nbf * nbf) for _ in range(3)]

    def context():
        eng = bd.Engine(s, bd.DONOF_RI_FP64)
        eng.transform(C, bd.DONOF_RI_HALF)
        bd.donof_ri_sync(eng.ctx)
        return eng

    eng = context()
    bd.donof_ri_apply_rotation(eng.ctx, k, out[0])
    eng.close()
    eng = context()
    with _LittleMemory(36 * MB):
        bd.donof_ri_apply_rotation(eng.ctx, k, out[1])
    eng.close()
    np.testing.assert_array_equal(out[1], out[0])
    eng = context()
    with _LittleMemory(28 * MB):  # the scratch and not even one piece: refused, the orbitals as they were
        with pytest.raises(bd.DonofError) as e:
            bd.donof_ri_apply_rotation(eng.ctx, k, out[2])
        assert e.value.status == bd.DONOF_RI_E_OOM
    bd.donof_ri_apply_rotation(eng.ctx, k, out[2])
    eng.close()
    np.testing.assert_array_equal(out[2], out[0])
