"""Contexts of different sizes beside one another: what one of them sets up for a kernel must not
take anything from another's launches, made later on one thread or at the same time on two.
Results are compared bit for bit with those of a context alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synthetic import draw_gamma, make_system, random_orthogonal, without_basis_functions  # noqa: E402


def _system(n_c, nbf, naux=70):
    full = make_system("ring", n_c=n_c, seed=6, n_weak_per=1)
    return without_basis_functions(full, full.nbf - nbf, full.naux - naux)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_a_larger_context_still_runs_after_a_smaller_one_is_made(prec):
    from paper_2012_15662_gb300 import binding as bd
    big, small = (make_system("ring", n_c=6, seed=6, n_weak_per=4), make_system("square"))
    rng = np.random.default_rng(1)
    C = [random_orthogonal(s.nbf, rng) for s in (big, small)]
    gamma = [draw_gamma(s.n_strong, s.n_weak_per, rng) for s in (big, small)]

    def run(eng, k):
        eng.transform(C[k], bd.DONOF_RI_FULL)
        J, K = eng.jk_mo()
        eng.jk_ao(want=False)
        E, lam = eng.energy_lagrangian(gamma[k])
        occ = eng.optimize_occupations(gamma[k], max_iter=3)
        return J, K, E, lam, occ[0], occ[1]

    engines = [bd.Engine(big, prec)]
    ref = run(engines[0], 0)
    engines.append(bd.Engine(small, prec))
    run(engines[1], 1)
    for a, b in zip(run(engines[0], 0), ref):
        np.testing.assert_array_equal(a, b)
    for e in engines:
        e.close()


@pytest.mark.parametrize("graph", [False, True])
def test_two_contexts_in_turn(graph):
    """Digits of J^(q), K^(q) at 48 and at 240 functions: 10 and 227 KB of shared memory."""
    import torch
    from paper_2012_15662_gb300 import binding as bd
    dev = torch.device("cuda", 0)
    runs, refs = [], []
    for n_c, nbf in ((10, 240), (3, 48)):
        s = _system(n_c, nbf)
        rng = np.random.default_rng(nbf)
        C = torch.tensor(random_orthogonal(nbf, rng), device=dev)
        g = torch.tensor(draw_gamma(s.n_strong, s.n_weak_per, rng), device=dev)
        stream = torch.cuda.Stream(device=dev)
        eng = bd.Engine(s, bd.DONOF_RI_SLICE4, stream=stream.cuda_stream)
        out = torch.zeros(nbf * nbf + 1, dtype=torch.float64, device=dev)
        torch.cuda.synchronize()

        def run(eng=eng, C=C, g=g, out=out, nbf=nbf):
            bd.donof_ri_iteration(eng.ctx, C, g, bd.DONOF_RI_HALF, None, None, out[nbf * nbf:], out[:nbf * nbf],
                                  use_graph=graph)
            bd.donof_ri_sync(eng.ctx)
            return out.cpu().numpy().copy()

        runs.append((run, eng))
        refs.append(run())
    for _ in range(3):
        for (run, _), ref in zip(runs, refs):
            np.testing.assert_array_equal(run(), ref)
    for _, eng in runs:
        eng.close()


@pytest.mark.parametrize("call", ["jk_ao", "occupations", "flambda"])
def test_two_contexts_on_two_threads(call):
    """A thread with a small context calls without a pause while another's launches need most of
    an SM's shared memory; each call must be accepted every time."""
    import torch
    from paper_2012_15662_gb300 import binding as bd
    sizes = ((10, 240), (3, 48)) if call == "jk_ao" else ((6, 144), (5, 120)) if call == "occupations" else ((6, 144), (3, 24))
    weak = 4 if call == "occupations" else 1
    engines, args = [], []
    for n_c, nbf in sizes:
        full = make_system("ring", n_c=n_c, seed=6, n_weak_per=weak)
        s = without_basis_functions(full, full.nbf - nbf, full.naux - 70)
        rng = np.random.default_rng(nbf)
        eng = bd.Engine(s, bd.DONOF_RI_SLICE4 if call == "jk_ao" else bd.DONOF_RI_FP64, stream=torch.cuda.Stream().cuda_stream)
        C, gamma = random_orthogonal(nbf, rng), draw_gamma(s.n_strong, s.n_weak_per, rng)
        eng.transform(C, bd.DONOF_RI_FULL)
        engines.append(eng)
        args.append((C, gamma))

    def once(k):
        eng, (C, gamma) = engines[k], args[k]
        if call == "jk_ao":
            eng.jk_ao(want=False)
        elif call == "occupations":
            eng.optimize_occupations(gamma, max_iter=0)
        else:
            eng.transform(C, bd.DONOF_RI_HALF)
            eng.jk_ao(want=False)
            eng.energy_lagrangian(gamma)
            bd.donof_ri_flambda_step(eng.ctx, None, True, 0.1)

    refused, done = [], threading.Event()

    def work(k, n):
        try:
            for _ in range(n):
                once(k)
                if k and done.is_set():
                    break
        except bd.DonofError as e:
            refused.append((k, str(e)))
        if k == 0:
            done.set()

    n = {"jk_ao": 2000, "occupations": 300, "flambda": 20}[call]
    threads = [threading.Thread(target=work, args=(0, n)), threading.Thread(target=work, args=(1, 10**9))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    for e in engines:
        bd.donof_ri_sync(e.ctx)
        e.close()
    assert not refused
