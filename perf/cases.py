"""The work that a user of the engine has it do, as cases to be timed.

Every case goes through the binding of the C ABI (`paper_2012_15662_gb300.binding`),
on the seeded CnH2n rings (and the four-atom square) that the tests, the drivers and
the benchmark use; `drop_bf` / `drop_aux` take functions off the end of the basis
and of the auxiliary set, which gives the odd and ragged sizes.

Kinds of pass
  iteration    one whole PNOF7 iteration on device buffers, replayed as a graph:
               the benchmark's step, and a program that keeps C and gamma on the GPU
  step         the orbital step of the solvers: half transform of device orbitals,
               J^(q), K^(q), energy and Lagrangian read back to the host
  contracted   the same quantities without J^(q), K^(q): full transform, J, K and the
               contracted Lagrangian
  occupations  twenty iterations of the occupation optimiser from the standard
               angles, for fixed orbitals (the optimiser's path is still determined to
               the last digits there; a whole optimisation repeats this)
  rotation     the line search's move of the quasi-Newton orbital step: back to the
               accepted orbitals, then C <- C expm(kappa), read back to the host
  setup        a new molecule: integrals, metric, fit, working basis, and its first
               J, K (the data generation of the learned start does this per ring)
"""
import numpy as np
import torch

from paper_2012_15662_gb300 import binding as bd
from synthetic import draw_gamma, make_system, pairing_columns, random_orthogonal, standard_gamma
from synthetic import without_basis_functions

PRECISIONS = {"fp64": bd.DONOF_RI_FP64, "tf32x3": bd.DONOF_RI_TF32X3, "slice4": bd.DONOF_RI_SLICE4}


def _case(name, kind, n_c, precision="slice4", mode="full", weak=4, drop_bf=0, drop_aux=0):
    c = dict(kind=kind, n_c=n_c, precision=precision, mode=mode, weak=weak, drop_bf=drop_bf, drop_aux=drop_aux)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest system of the tests: launches and latency
        _case("square4_iteration", "iteration", 0),
        # a small ring, where most inner iterations of a study are spent
        _case("c6h12_iteration", "iteration", 6),
        # the solvers' orbital step on an ordinary ring
        _case("c10h20_step", "step", 10, mode="half"),
        # every tile edge ragged (nbf 229, naux 811)
        _case("ragged_iteration", "iteration", 10, drop_bf=11, drop_aux=29),
        # the largest small-basis sizes: K = nbf in one chunk, several chunks over naux
        _case("c16h32_iteration", "iteration", 16),
        # the headline workload
        _case("c20h40_iteration", "iteration", 20),
        # the contracted Lagrangian, odd basis (nbf 471, naux 1680)
        _case("c16h32_contracted", "contracted", 16, drop_bf=9),
        # the plain FP64 form, against which the others are judged and which the
        # exact restart and the training data use
        _case("c6h12_fp64_iteration", "iteration", 6, precision="fp64"),
        # the split-TF32 form
        _case("c10h20_tf32x3_iteration", "iteration", 10, precision="tf32x3"),
        # the occupation optimiser at 400 orbitals (few auxiliary functions: it only
        # sees J and K)
        _case("occupations_400", "occupations", 20, precision="fp64", drop_aux=2400),
        # the quasi-Newton rotation at 720 functions (few auxiliary functions: it only
        # sees the orbitals)
        _case("rotation_720", "rotation", 20, mode="half", drop_aux=2488),
        # a new context for an ordinary ring
        _case("c10h20_setup", "setup", 10),
    ]


def draw(rng):
    kind = rng.choice(["iteration"] * 5 + ["step", "step", "contracted", "occupations", "rotation", "setup"])
    few_aux = kind in ("occupations", "rotation")
    precision = "slice4"
    if kind == "occupations":
        precision = "fp64"
    elif kind in ("iteration", "step", "setup"):
        precision = rng.choice(["slice4"] * 6 + ["tf32x3", "fp64"])
    largest = {"iteration": 20, "step": 20, "contracted": 16, "occupations": 20, "rotation": 20, "setup": 12}[kind]
    if precision == "fp64" and not few_aux:
        largest = 7
    if precision == "tf32x3":
        largest = 12
    # spread over the logarithm of the ring's size
    n_c = int(round(3.0 * (largest / 3.0) ** rng.random()))
    weak = rng.choice([4, 4, 4, 3, 2, 1])
    nbf, naux = (24, 84) if n_c <= 12 else ((30, 105) if n_c <= 16 else (36, 126))
    spare = n_c * nbf - 4 * n_c * (1 + weak)
    drop_bf = rng.randint(0, min(spare, 2 * n_c + 1))
    drop_aux = rng.randint(n_c * naux - 136, n_c * naux - 40) if few_aux else rng.randint(0, 5 * n_c)
    mode = "half" if kind in ("step", "rotation") else "full"
    if kind == "iteration":
        mode = rng.choice(["full", "full", "half"])
    return _case(None, kind, n_c, precision, mode, weak, drop_bf, drop_aux)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _system(case, seed):
    if case["n_c"] == 0:
        s = make_system("square")
    else:
        s = make_system("ring", n_c=case["n_c"], seed=seed, n_weak_per=case["weak"])
    if case["drop_bf"] or case["drop_aux"]:
        s = without_basis_functions(s, case["drop_bf"], case["drop_aux"])
    return s


def _norm_s(a):
    return (2.0 * a / np.pi) ** 0.75


def _overlap(s):
    X, a = s.atom_xyz[s.bf_atom], s.bf_alpha
    p = a[:, None] + a[None, :]
    r2 = ((X[:, None, :] - X[None, :, :]) ** 2).sum(-1)
    return (_norm_s(a)[:, None] * _norm_s(a)[None, :]) * (np.pi / p) ** 1.5 * np.exp(-(a[:, None] * a[None, :] / p) * r2)


def _inputs(case, seed):
    """The molecule, S-orthonormal orbitals C = S^-1/2 Q, the angles and a rotation generator."""
    s = _system(case, seed)
    rng = np.random.default_rng(50_000 + seed)
    S = _overlap(s)
    ev, U = np.linalg.eigh(S)
    C = (U * ev ** -0.5) @ (U.T @ random_orthogonal(s.nbf, rng))
    gamma = draw_gamma(s.n_strong, s.n_weak_per, rng)
    kappa = None
    if case["kind"] == "rotation":
        # a step of up to 0.2 radians in any pair, as the line search takes them
        a = np.tril(rng.standard_normal((s.nbf, s.nbf)), -1)
        kappa = a - a.T
        kappa = np.ascontiguousarray(0.2 / np.abs(kappa).max() * kappa)
    return s, S, np.ascontiguousarray(C), gamma, kappa


_streams = {}


def _stream():
    """The program's one work stream (graphs need a stream of their own)."""
    if "s" not in _streams:
        _streams["s"] = torch.cuda.Stream()
    return _streams["s"].cuda_stream


class _State:
    """A context and the buffers a program keeps with it; the context goes when the state does."""

    def __init__(self, case, seed):
        s, _, C, gamma, kappa = _inputs(case, seed)
        self.case, self.system = case, s
        nb, m = s.nbf, s.n_omega
        f8 = dict(dtype=torch.float64, device="cuda")
        self.C_host = np.ascontiguousarray(C.T)  # the ABI's column-major buffer
        self.gamma_host = gamma
        self.kappa = kappa
        self.eng = None
        kind = case["kind"]
        if kind == "setup":
            self.C_mu_p = C
            return
        self.eng = bd.Engine(s, PRECISIONS[case["precision"]], stream=_stream())
        self.C = torch.tensor(self.C_host.reshape(-1), **f8)
        self.gamma = torch.tensor(gamma, **f8)
        self.mode = bd.DONOF_RI_FULL if case["mode"] == "full" else bd.DONOF_RI_HALF
        if kind in ("iteration", "contracted"):
            self.J, self.K = torch.empty(m, m, **f8), torch.empty(m, m, **f8)
            if self.mode == bd.DONOF_RI_HALF:
                self.J = self.K = None
            self.E, self.lam = torch.empty(1, **f8), torch.empty(nb, nb, **f8)
        elif kind == "step":
            self.E, self.lam = np.zeros(1), np.empty((nb, nb))
        elif kind == "rotation":
            self.C_out = np.empty((nb, nb))
        elif kind == "occupations":
            self.gamma0 = standard_gamma(s.n_strong, s.n_weak_per)
            bd.donof_ri_transform(self.eng.ctx, self.C, bd.DONOF_RI_FULL)
        torch.cuda.synchronize()


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    kind = state.case["kind"]
    if kind == "setup":
        eng = bd.Engine(state.system, PRECISIONS[state.case["precision"]], stream=_stream())
        eng.transform(state.C_mu_p, bd.DONOF_RI_FULL)
        J, K = eng.jk_mo()
        eng.close()
        return {"J": J, "K": K}
    ctx = state.eng.ctx
    if kind == "iteration":
        bd.donof_ri_iteration(ctx, state.C, state.gamma, state.mode, state.J, state.K, state.E, state.lam)
        out = {"E": state.E, "lambda": state.lam}
        if state.J is not None:
            out.update(J=state.J, K=state.K)
        return out
    if kind == "step":
        bd.donof_ri_transform(ctx, state.C, state.mode)
        bd.donof_ri_jk_ao_batch(ctx)
        bd.donof_ri_energy_lagrangian(ctx, state.gamma_host, state.E, state.lam)
        return {"E": state.E, "lambda": state.lam}
    if kind == "contracted":
        bd.donof_ri_transform(ctx, state.C, state.mode)
        bd.donof_ri_jk_mo(ctx, state.J, state.K)
        bd.donof_ri_energy_lagrangian_contracted(ctx, state.gamma, state.E, state.lam)
        return {"E": state.E, "lambda": state.lam, "J": state.J, "K": state.K}
    if kind == "occupations":
        gamma, E, grad, iterations, reason = state.eng.optimize_occupations(state.gamma0, max_iter=20, gtol=1e-8,
                                                                            etol=1e-14)
        return {"gamma": gamma, "E": E, "gradient": grad, "iterations": iterations, "reason": reason}
    if kind == "rotation":
        bd.donof_ri_transform(ctx, state.C, state.mode)
        bd.donof_ri_apply_rotation(ctx, state.kappa, state.C_out)
        return {"C": state.C_out}
    raise ValueError(kind)


def work(case):
    """Multiplications and additions of the algorithm (symmetric halves once), and bytes:
    the fitted tensor (its symmetric half, 8 bytes an element) and the orbitals read once,
    the results written once."""
    s = _system(case, 1)
    nb, nx, m = s.nbf, s.naux, s.n_omega
    tensor = 8.0 * nx * nb * (nb + 1) / 2
    half = 2.0 * nb * nb * nx * m
    full = 2.0 * nb * nx * m * m + float(nx) * m * (m + 1)
    orbital = 2.0 * nb * (nb + 1) * nx * m + 4.0 * nb * nb * m * m
    contracted = 4.0 * nb * nx * m * m + 2.0 * nx * m * m + 4.0 * nb * nb * m
    kind = case["kind"]
    full = full if case["mode"] == "full" else 0.0
    if kind == "occupations":
        # about 27 evaluations, 20 operations per pair
        return {"bytes": 16.0 * m * m, "flops": 27 * 20.0 * m * m}
    if kind == "rotation":
        # a series of at least five products, a few squarings, the orbitals and their metric
        return {"bytes": tensor + 24.0 * nb * nb, "flops": 24.0 * nb ** 3 + half}
    if kind == "setup":
        fit = nx ** 3 / 3.0 + float(nx) * nx * nb * (nb + 1) / 2
        return {"bytes": tensor + 8.0 * nx * nx + 16.0 * m * m, "flops": fit + half + full}
    out = 8.0 * (nb * nb + 1) + (16.0 * m * m if full else 0.0)
    return {"bytes": tensor + 8.0 * nb * nb + out, "flops": half + full + (contracted if kind == "contracted" else orbital)}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch / numpy
# ---------------------------------------------------------------------------
def _boys(t):
    ts = torch.clamp(t, min=1e-8)
    big = 0.5 * torch.sqrt(np.pi / ts) * torch.erf(torch.sqrt(ts))
    return torch.where(t < 1e-8, 1.0 - t / 3.0 + t * t / 10.0, big)


def _integrals(s):
    """H, E_nuc and the fitted tensor B[P][mu][nu] (G = L L^T, B = L^-1 (P|mu nu)) on the GPU."""
    f8 = dict(dtype=torch.float64, device="cuda")
    xyz, Z = torch.tensor(s.atom_xyz, **f8), torch.tensor(s.atom_charge, **f8)
    X, a = torch.tensor(s.atom_xyz[s.bf_atom], **f8), torch.tensor(s.bf_alpha, **f8)
    Y, c = torch.tensor(s.atom_xyz[s.aux_atom], **f8), torch.tensor(s.aux_alpha, **f8)
    p = a[:, None] + a[None, :]
    mu = a[:, None] * a[None, :] / p
    r2 = ((X[:, None, :] - X[None, :, :]) ** 2).sum(-1)
    kab = torch.exp(-mu * r2) * ((2.0 * a / np.pi) ** 0.75)[:, None] * ((2.0 * a / np.pi) ** 0.75)[None, :]
    P = (a[:, None, None] * X[:, None, :] + a[None, :, None] * X[None, :, :]) / p[..., None]
    S = (np.pi / p) ** 1.5 * kab
    H = mu * (3.0 - 2.0 * mu * r2) * S
    for z, x in zip(Z, xyz):
        H = H - z * (2.0 * np.pi / p) * kab * _boys(p * ((P - x) ** 2).sum(-1))
    enuc = 0.0
    q, w = s.atom_xyz, s.atom_charge
    for i in range(len(w)):
        for j in range(i):
            enuc += w[i] * w[j] / np.linalg.norm(q[i] - q[j])
    two = 2.0 * np.pi ** 2.5
    nc = (2.0 * c / np.pi) ** 0.75 * torch.sqrt(c / (4.0 * np.pi))
    cc = c[:, None] + c[None, :]
    G = nc[:, None] * nc[None, :] * two / (c[:, None] * c[None, :] * torch.sqrt(cc))
    G = G * _boys(c[:, None] * c[None, :] / cc * ((Y[:, None, :] - Y[None, :, :]) ** 2).sum(-1))
    nb, nx = s.nbf, s.naux
    B = torch.empty(nx, nb * nb, **f8)
    for k in range(nx):
        t = p * c[k] / (p + c[k]) * ((P - Y[k]) ** 2).sum(-1)
        B[k] = (nc[k] * two / (p * c[k] * torch.sqrt(p + c[k])) * kab * _boys(t)).reshape(-1)
    B = torch.linalg.solve_triangular(torch.linalg.cholesky(G), B, upper=False)
    return S, H, float(enuc), B.reshape(nx, nb, nb)


def _occupations(gamma, s):
    """n_p and the map's pieces: alpha [N_I][N_g] and d alpha_i / d w_j."""
    NI, Ng = s.n_strong, s.n_weak_per
    cg = np.cos(gamma[:NI]) ** 2
    n_s, h = 0.5 * (1.0 + cg), 1.0 - 0.5 * (1.0 + cg)
    w = gamma[NI:].reshape(NI, Ng - 1)
    alpha, dalpha = np.empty((NI, Ng)), np.zeros((NI, Ng, max(Ng - 1, 0)))
    for i in range(Ng):
        tail = np.cos(w[:, i]) ** 2 if i < Ng - 1 else np.ones(NI)
        alpha[:, i] = np.prod(np.sin(w[:, :i]) ** 2, axis=1) * tail
        for j in range(i):
            rest = [k for k in range(i) if k != j]
            dalpha[:, i, j] = np.prod(np.sin(w[:, rest]) ** 2, axis=1) * np.sin(2.0 * w[:, j]) * tail
        if i < Ng - 1:
            dalpha[:, i, i] = -np.prod(np.sin(w[:, :i]) ** 2, axis=1) * np.sin(2.0 * w[:, i])
    sub, rank = pairing_columns(NI, Ng)
    n = np.where(rank < 0, n_s[sub], h[sub] * alpha[sub, np.maximum(rank, 0)])
    return n, h, alpha, dalpha, sub, rank


def _couplings(n, sub, rank):
    same = sub[:, None] == sub[None, :]
    root = np.sqrt(n[:, None] * n[None, :])
    phi = np.sqrt(n * (1.0 - n))
    strong = (rank[:, None] < 0) | (rank[None, :] < 0)
    A = np.where(same, 0.0, 2.0 * n[:, None] * n[None, :])
    Bc = np.where(same, np.where(strong, root, -root), n[:, None] * n[None, :] + phi[:, None] * phi[None, :])
    np.fill_diagonal(A, n)
    np.fill_diagonal(Bc, 0.0)
    return A, Bc


def _minimise(gamma, s, Hd, J, K, enuc, max_iter, gtol, etol):
    """L-BFGS (8 pairs, backtracking to sufficient decrease 1e-4) on E(gamma): the optimiser's own rules."""
    def evaluate(x):
        n, h, alpha, dalpha, sub, rank = _occupations(x, s)
        same = sub[:, None] == sub[None, :]
        sign = np.where((rank[:, None] < 0) | (rank[None, :] < 0), 1.0, -1.0)
        Ks, Jo, Ko = np.where(same, sign * K, 0.0), np.where(same, 0.0, J), np.where(same, 0.0, K)
        np.fill_diagonal(Ks, 0.0)
        root, phi = np.sqrt(n), np.sqrt(n * (1.0 - n))
        inv = np.divide(1.0, root, out=np.zeros_like(root), where=root > 0)
        dphi = np.divide(1.0 - 2.0 * n, 2.0 * phi, out=np.zeros_like(phi), where=phi > 0)
        v = 2.0 * Hd + np.diag(J) - inv * (Ks @ root) + 4.0 * (Jo @ n) - 2.0 * (Ko @ n) - 2.0 * dphi * (Ko @ phi)
        E = enuc + 2.0 * n @ Hd + n @ np.diag(J) - root @ (Ks @ root) + 2.0 * n @ (Jo @ n) - n @ (Ko @ n) - phi @ (Ko @ phi)
        D = np.empty((s.n_strong, s.n_weak_per + 1))
        D[sub, rank + 1] = v
        dh = 0.5 * np.sin(2.0 * x[:s.n_strong])
        gs = dh * ((alpha * D[:, 1:]).sum(1) - D[:, 0])
        gw = h[:, None] * np.einsum("gij,gi->gj", dalpha, D[:, 1:])
        return E, np.concatenate([gs, gw.reshape(-1)])

    x = np.array(gamma)
    E, g = evaluate(x)
    pairs, it, reason = [], 0, 1
    for it in range(max_iter):
        gmax = np.abs(g).max()
        if gmax <= gtol:
            return x, E, g, it, 0
        d, al = g.copy(), []
        for sk, yk in reversed(pairs):
            al.append((sk @ d) / (sk @ yk))
            d -= al[-1] * yk
        d *= (pairs[-1][0] @ pairs[-1][1]) / (pairs[-1][1] @ pairs[-1][1]) if pairs else min(1.0, 0.5 / gmax)
        for (sk, yk), ak in zip(pairs, reversed(al)):
            d += (ak - (yk @ d) / (sk @ yk)) * sk
        d = -d
        if not g @ d < 0.0:
            pairs, d = [], -min(1.0, 0.5 / gmax) * g
        slope, t = g @ d, 1.0
        for _ in range(40):
            xn = x + t * d
            En, gn = evaluate(xn)
            if En <= E + 1e-4 * t * slope:
                break
            t *= 0.5
        else:
            return x, E, g, it, 2
        if (xn - x) @ (gn - g) > 0.0:
            pairs = (pairs + [(xn - x, gn - g)])[-8:]
        drop, x, E, g = E - En, xn, En, gn
        if drop <= etol * max(1.0, abs(E)):
            return x, E, g, it + 1, 3
    return x, E, g, max_iter, reason


def exact(case, seed):
    s, S_np, C_np, gamma, kappa = _inputs(case, seed)
    nb, m = s.nbf, s.n_omega
    f8 = dict(dtype=torch.float64, device="cuda")
    kind = case["kind"]
    if kind == "rotation":
        C = torch.tensor(C_np, **f8) @ torch.linalg.matrix_exp(torch.tensor(kappa, **f8))
        return {"C": C.T.contiguous().cpu().numpy()}
    S, H, enuc, B = _integrals(s)
    C = torch.tensor(C_np, **f8)
    Co = C[:, :m]
    bh = torch.matmul(Co.T, B)  # [P][p][nu]
    del B
    d = (bh * Co.T).sum(-1)  # [P][p]
    K, Y = torch.zeros(m, m, **f8), torch.zeros(nb, m, **f8)
    want_lambda = kind in ("iteration", "step", "contracted")
    if want_lambda:
        n, _, _, _, sub, rank = _occupations(gamma, s)
        A, Bc = (torch.tensor(v, **f8) for v in _couplings(n, sub, rank))
        n = torch.tensor(n, **f8)
        w = d @ A  # [P][p]
        Y = (H @ Co) * n + torch.einsum("Pp,Ppm->mp", w, bh)
    for P0 in range(0, s.naux, 64):
        b = bh[P0:P0 + 64]
        bf = torch.matmul(b, Co)  # b^P_qp
        K += (bf * bf).sum(0)
        if want_lambda:
            Y -= torch.matmul(b.transpose(1, 2), bf * Bc).sum(0)
    J = d.T @ d
    if kind == "setup":
        return {"J": J.cpu().numpy(), "K": K.cpu().numpy()}
    Hd = (Co * (H @ Co)).sum(0)
    if kind == "occupations":
        x, E, g, it, reason = _minimise(standard_gamma(s.n_strong, s.n_weak_per), s, Hd.cpu().numpy(), J.cpu().numpy(),
                                        K.cpu().numpy(), enuc, 20, 1e-8, 1e-14)
        sn, cs = np.sin(x), np.cos(x)
        return {"gamma": np.arctan2(np.abs(sn), np.abs(cs)), "E": float(E), "gradient": np.where(sn * cs < 0.0, -g, g),
                "iterations": it, "reason": reason}
    lam = torch.zeros(nb, nb, **f8)
    lam[:m] = (C.T @ Y).T  # row p holds lambda_qp over q, the ABI's column-major layout
    E = enuc + float((n * Hd).sum() + torch.diagonal(lam)[:m].sum())
    out = {"E": E, "lambda": lam}
    if kind == "iteration":
        out["E"] = torch.tensor([E], **f8)
        if case["mode"] == "full":
            out.update(J=J, K=K)
    elif kind == "contracted":
        out.update(E=torch.tensor([E], **f8), J=J, K=K)
    else:
        out.update(E=np.array([E]), **{"lambda": lam.cpu().numpy()})
    return out
