"""The work that users of the library have it do: one case per call that a program makes, from the smallest molecule
to the 180-function workload, with the inputs that such a program holds and the same results in plain 64-bit torch.

Sizes are those of the workloads in ``synth.py``, of the tests and of the benchmark.  A case names the call (``kind``),
the molecule (atoms, basis, primitives per shell), the method's orders (n, P, omega) and the options of the call; the
molecule, the densities and the orbitals are drawn from the seed.
"""
import math

import numpy as np
import torch

from paper_2210_13069_gb300 import lrtei, synth

DEV = "cuda" if torch.cuda.is_available() else "cpu"
SHELLS = {"spd": (("s", 3), ("p", 2), ("d", 1)), "s": (("s", 5),)}  # shells of one atom
NBF = {"spd": 15, "s": 5}                                           # their functions


def listed():
    return [
        # The headline call: the full B of the 180-function molecule, plan resident, default tensor-core precision.
        dict(name="b_nb180", kind="b", atoms=12, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="split_f16"),
        # One small molecule at odd orders, as in a scan over many of them: launches and ragged tiles count.
        dict(name="b_nb45_ragged", kind="b", atoms=3, basis="spd", nprim=3, n=13, P=11, omega=0.5, prec="split_f16"),
        # An uncontracted basis, which the library assembles by Algorithm 1 (Hadamard form).
        dict(name="b_nb180_uncontracted", kind="b", atoms=12, basis="spd", nprim=1, n=24, P=32, omega=0.4, prec="split_f16"),
        # The default precision of a Plan: a reference B in FP64.
        dict(name="b_nb60_fp64", kind="b", atoms=4, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="fp64"),
        # The Khatri-Rao compressed plan with the precise (eight-product) scheme.
        dict(name="b_nb180_compressed", kind="b", atoms=12, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="split_f16_8",
             eps=1e-8),
        # Adaptive boxes: partition blocks of B with one coefficient block per pair of boxes.
        dict(name="b_nb60_adaptive", kind="b", atoms=4, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="split_f16",
             parts=4),
        # A molecule seen once (a geometry scan): plan from host arrays, B, plan destroyed.
        dict(name="first_b_nb120", kind="first", atoms=8, basis="spd", nprim=3, n=20, P=28, omega=0.33, prec="split_f16"),
        # J-builds inside an SCF or response iteration: 32 densities, operands and buffers resident.
        dict(name="j_nb180_r32", kind="j", atoms=12, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="split_f16", R=32),
        # The same in the default precision.
        dict(name="j_nb120_fp64", kind="j", atoms=8, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="fp64", R=16),
        # The smallest call: one density of the 20-function molecule.
        dict(name="j_nb20_r1_fp64", kind="j", atoms=4, basis="s", nprim=1, n=16, P=20, omega=0.5, prec="fp64", R=1),
        # Many molecules of uneven size in one call.
        dict(name="j_batch8", kind="batch", mols=8, atoms=12, R=16, prec="split_f16"),
        # Long-range exchange of a hybrid functional: half as many orbitals as functions.
        dict(name="x_nb180", kind="x", atoms=12, basis="spd", nprim=3, n=24, P=32, omega=0.4, prec="split_f16", orbs=90),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds, sizes spread over their logarithm, at most the work of the listed one of its kind."""
    like = rng.choice(listed())
    most = work(like)
    for _ in range(10000):
        c = {k: v for k, v in like.items() if k != "name"}
        c["atoms"] = _log_int(rng, 1 if c["kind"] == "j" else 2, like["atoms"])
        if c["kind"] == "batch":
            c["mols"] = rng.randint(2, like["mols"])
            c["atoms"] = rng.randint(3, like["atoms"])
        else:
            c["n"] = rng.randint(11, 28)
            c["P"] = rng.randint(11, 40)
            c["omega"] = rng.choice([0.2, 0.33, 0.4, 0.5, 1.0])
        if "R" in c:
            c["R"] = _log_int(rng, 1, 48)
        if "orbs" in c:
            c["orbs"] = _log_int(rng, 1, NBF[c["basis"]] * c["atoms"] // 2)
        if "parts" in c:
            c["parts"] = rng.randint(2, 4)
        if "eps" in c:
            c["eps"] = rng.choice([1e-6, 1e-7, 1e-8])
        w = work(c)
        if w["flops"] <= most["flops"] and w["bytes"] <= most["bytes"]:
            return c
    return {k: v for k, v in like.items() if k != "name"}


def _molecule(case, seed):
    if case["basis"] == "s":
        return synth.random_molecule(seed, natoms=case["atoms"], cube=6.0, shells_per_atom=SHELLS["s"], nprim=case["nprim"],
                                     alpha_range=(0.1, 50.0), omega=case["omega"], n=case["n"], P=case["P"])
    return synth.workload_spd(seed, natoms=case["atoms"], cube=12.0 * (case["atoms"] / 12.0) ** (1.0 / 3.0),
                              omega=case["omega"], n=case["n"], P=case["P"], nprim=case["nprim"])


def _batch(case, seed):
    """Molecules of the batched workload's recipe: sizes fixed by the case, geometry and basis by the seed."""
    rng = np.random.Generator(np.random.Philox(77 + case["mols"]))
    mols = []
    for i in range(case["mols"]):
        c = dict(atoms=int(rng.integers(2, case["atoms"] + 1)), basis="spd", nprim=3,
                 omega=float(rng.choice([0.2, 0.33, 0.5, 1.0])), n=int(rng.integers(20, 26)), P=int(rng.integers(24, 41)))
        mols.append((c, None if seed is None else _molecule(c, seed * 100 + i)))
    return mols


def _densities(seed, nbf, R):
    """R symmetric positive densities X X^T, as synth.random_densities, drawn on the device."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
    X = torch.randn((R, nbf, max(1, nbf // 4)), generator=g, device=DEV, dtype=torch.float64) / math.sqrt(nbf)
    D = X @ X.transpose(1, 2)
    return (0.5 * (D + D.transpose(1, 2))).contiguous()


def _orbitals(seed, nbf, orbs):
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 9)
    return torch.randn((orbs, nbf), generator=g, device=DEV, dtype=torch.float64) / math.sqrt(nbf)


def prepare(case, seed):
    if case["kind"] == "batch":
        mols = [m for _, m in _batch(case, seed)]
        D = [_densities(seed + i, m.nbf, case["R"]) for i, m in enumerate(mols)]
        return {"case": case, "plans": [lrtei.Plan(m, case["prec"]) for m in mols], "D": D,
                "out": [torch.empty_like(d) for d in D]}
    mol = _molecule(case, seed)
    nbf = mol.nbf
    state = {"case": case, "mol": mol}
    if case["kind"] == "first":
        state["out"] = torch.empty((nbf * nbf, nbf * nbf), dtype=torch.float64, device="cuda")
        return state
    plan = lrtei.Plan(mol, case["prec"], adaptive=(1e-20, case["parts"]) if "parts" in case else None)
    if "eps" in case:
        plan.compress(case["eps"])
    state["plan"] = plan
    if case["kind"] == "b":
        state["out"] = torch.empty((nbf * nbf, nbf * nbf), dtype=torch.float64, device="cuda")
    elif case["kind"] == "j":
        state["D"] = _densities(seed, nbf, case["R"])
        state["out"] = torch.empty_like(state["D"])
    else:
        state["Q"] = _orbitals(seed, nbf, case["orbs"])
        state["out"] = torch.empty((nbf, nbf), dtype=torch.float64, device="cuda")
    return state


def run(state):
    kind = state["case"]["kind"]
    if kind == "b":
        return state["plan"].assemble_B(out=state["out"])
    if kind == "first":
        plan = lrtei.Plan(state["mol"], state["case"]["prec"])
        plan.assemble_B(out=state["out"])
        plan.close()
        return state["out"]
    if kind == "j":
        return state["plan"].jbuild(state["D"], out=state["out"])
    if kind == "x":
        return state["plan"].exchange(state["Q"], out=state["out"])
    lrtei.lrtei_jbuild_batched([p.plan for p in state["plans"]], state["D"], [d.shape[0] for d in state["D"]], state["out"])
    return state["out"]


def work(case):
    """Inputs (moments and coefficients of the plan, densities or orbitals) read once, the result written once; the
    multiplications and additions of the cheaper form of Theorem 1 on unique pairs, the Chebyshev coefficients' zeros
    (odd total degree) left out."""
    if case["kind"] == "batch":
        parts = [work(dict(c, kind="j", R=case["R"])) for c, _ in _batch(case, None)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nbf, n, P = NBF[case["basis"]] * case["atoms"], case["n"], case["P"]
    npair = nbf * (nbf + 1) // 2
    rows = npair * case["nprim"] ** 2
    n3, node = float(n) ** 3, 3.0 * P * float(n) ** 4  # node: K applied to one vector of n^3 by mode products
    bytes_ = 8.0 * (3 * rows * n + 3 * P * n * n)
    if case["kind"] in ("b", "first"):
        factored = npair * node * (case.get("parts", 1) + 1) / 2 + float(npair) ** 2 * n3
        hadamard = 0.5 * float(npair) ** 2 * P * case["nprim"] ** 4 * (6 * n + 3)
        return {"bytes": bytes_ + 8.0 * float(nbf) ** 4, "flops": min(factored, hadamard)}
    if case["kind"] == "j":
        return {"bytes": bytes_ + 16.0 * case["R"] * nbf * nbf, "flops": case["R"] * (4.0 * npair * n3 + node)}
    orbs = case["orbs"]
    return {"bytes": bytes_ + 8.0 * (orbs * nbf + nbf * nbf),
            "flops": orbs * (2.0 * nbf * nbf * n3 + nbf * node + float(nbf) * nbf * n3)}


# ---------------------------------------------------------------------------------------------------------------
# The same results in 64 bits: moments by a fine Gauss-Legendre rule, F and K as dense matrices, plain products.
# ---------------------------------------------------------------------------------------------------------------

def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _fact2(k):
    return 1.0 if k <= 1 else k * _fact2(k - 2)


def _chebyshev(n, u):
    T = [torch.ones_like(u), u]
    for _ in range(2, n):
        T.append(2 * u * T[-1] - T[-2])
    return torch.stack(T[:n], dim=-1)


class _Exact:
    """F (rows: unique pairs mu <= nu; columns: m1, m2, m3) and blocks of K of one molecule."""

    def __init__(self, mol, tau=0.0, parts=1):
        self.mol, self.n, self.P = mol, mol.n, mol.P
        sh = mol.shells
        func, coef = [], []  # (shell, powers) and normalised coefficients of every function
        for s, x in enumerate(sh):
            for lx in range(x.l, -1, -1):
                for ly in range(x.l - lx, -1, -1):
                    p = (lx, ly, x.l - lx - ly)
                    a = x.exps
                    norm = (2 * a / np.pi) ** 0.75 * (4 * a) ** (0.5 * x.l) / math.sqrt(
                        np.prod([_fact2(2 * q - 1) for q in p]))
                    ov = (2 * np.sqrt(np.outer(a, a)) / np.add.outer(a, a)) ** (x.l + 1.5)
                    func.append((s,) + p)
                    coef.append(x.coefs * norm / math.sqrt(x.coefs @ ov @ x.coefs))
        self.nbf = N = len(func)
        mu, nu = np.triu_indices(N)
        self.npair = len(mu)
        self.index = torch.zeros((N, N), dtype=torch.int64, device=DEV)
        r = torch.arange(self.npair, device=DEV)
        m_, n_ = torch.as_tensor(mu, device=DEV), torch.as_tensor(nu, device=DEV)
        self.index[m_, n_] = r
        self.index[n_, m_] = r
        self.mu, self.nu = m_, n_
        func, coef = np.array(func), np.array(coef)
        C = np.array([s.center for s in sh])
        E = np.array([s.exps for s in sh])
        lo, hi = C.min(0), C.max(0)
        centre = 0.5 * (lo + hi)
        s1, s2 = func[mu, 0], func[nu, 0]
        K = E.shape[1]
        if parts > 1:  # boxes by the support of each pair, about equal counts, equal supports together
            a, b = E[s1][:, :, None], E[s2][:, None, :]
            p = a + b
            Pc = (a[..., None] * C[s1][:, None, None] + b[..., None] * C[s2][:, None, None]) / p[..., None]
            sup = (np.abs(Pc - centre).max(-1) + np.sqrt(math.log(1 / tau) / p)).max((1, 2))
            order = np.argsort(sup, kind="stable")
            cuts = [0]
            for k in range(1, parts):
                c = max(cuts[-1], k * len(mu) // parts)
                while 0 < c < len(mu) and sup[order[c]] == sup[order[c - 1]]:
                    c += 1
                cuts.append(c)
            cuts.append(len(mu))
            groups = [order[cuts[k]:cuts[k + 1]] for k in range(parts) if cuts[k + 1] > cuts[k]]
            half = [float(sup[g].max()) for g in groups]
        else:
            groups = [np.arange(len(mu))]
            half = [float(np.max(0.5 * (hi - lo)) + math.sqrt(math.log(1e16) / (2 * E.min())))]
        self.groups, self.half = [torch.as_tensor(g, device=DEV) for g in groups], half
        box = np.zeros(len(mu))
        for g, h in zip(groups, half):
            box[g] = h
        # F in blocks of pairs
        n = self.n
        self.F = torch.empty((self.npair, n ** 3), dtype=torch.float64, device=DEV)
        x16, w16 = np.polynomial.legendre.leggauss(20)
        step = max(1, 3_000_000 // (K * K * 640))
        for p0 in range(0, self.npair, step):
            q = slice(p0, min(self.npair, p0 + step))
            a, b = _t(E[s1[q]])[:, :, None], _t(E[s2[q]])[:, None, :]
            c = (_t(coef[mu[q]])[:, :, None] * _t(coef[nu[q]])[:, None, :]).flatten(1)
            p = a + b
            S = []
            for d in range(3):
                A, B = _t(C[s1[q], d])[:, None, None], _t(C[s2[q], d])[:, None, None]
                Pc, pre = (a * A + b * B) / p, torch.exp(-a * b / p * (A - B) ** 2)
                bx = _t(box[q])[:, None, None]
                left = torch.maximum(Pc - 10 / p.sqrt(), centre[d] - bx)
                right = torch.maximum(left, torch.minimum(Pc + 10 / p.sqrt(), centre[d] + bx))
                cell = (right - left) / 32
                x = left[..., None, None] + cell[..., None, None] * (
                    torch.arange(32, device=DEV, dtype=torch.float64)[:, None] + 0.5 + 0.5 * _t(x16))
                x = x.flatten(3)
                w = (0.5 * cell[..., None] * _t(np.tile(w16, 32)))
                pa, pb = _t(func[mu[q], 1 + d])[:, None, None, None], _t(func[nu[q], 1 + d])[:, None, None, None]
                f = w * pre[..., None] * (x - A[..., None]) ** pa * (x - B[..., None]) ** pb * torch.exp(
                    -p[..., None] * (x - Pc[..., None]) ** 2)
                u = (x - centre[d]) / bx[..., None]
                # Chebyshev sums by recurrence, so that no array of points times orders is held
                T0, T1, m = torch.ones_like(u), u, []
                for k in range(n):
                    m.append((f * T0).sum(-1))
                    T0, T1 = T1, 2 * u * T1 - T0
                S.append(torch.stack(m, -1).flatten(1, 2))
            YZ = (S[1][..., :, None] * S[2][..., None, :]).flatten(2)
            self.F[q] = ((c[..., None] * S[0]).transpose(1, 2) @ YZ).flatten(1)

    def _K(self, hx, hy):
        """The blocks of K = (omega / sqrt(pi)) sum_p w_p A_p x A_p x A_p between boxes of half-widths hx and hy, by
        parity of the degrees (A_p(a, b) = 0 for odd a + b): [(row indices, matrix)]."""
        n, P, om = self.n, self.P, self.mol.omega
        z, w = np.polynomial.legendre.leggauss(P)
        s = _t(om * (1 + z) / 2)
        u = torch.cos((2 * torch.arange(1, n + 1, device=DEV, dtype=torch.float64) - 1) * math.pi / (2 * n))
        cT = _chebyshev(n, u) * torch.cat([_t([1.0]), _t(np.full(n - 1, 2.0))]) / n
        A = cT.T @ torch.exp(-(s[:, None, None] * (hx * u[:, None] - hy * u[None, :])) ** 2) @ cT
        m = torch.arange(n ** 3, device=DEV).reshape(n, n, n)
        W = _t(w * om / math.sqrt(math.pi))
        out = []
        for e in range(8):
            i, j, k = (torch.arange((e >> t) & 1, n, 2, device=DEV) for t in range(3))
            if min(len(i), len(j), len(k)) == 0:
                continue
            Ax, Ay, Az = (A[:, t[:, None], t[None, :]] for t in (i, j, k))
            L = (W[:, None, None] * Ax.flatten(1)[:, :, None] * Ay.flatten(1)[:, None, :]).flatten(1)
            Kb = (L.T @ Az.flatten(1)).reshape(len(i), len(i), len(j), len(j), len(k), len(k))
            Kb = Kb.permute(0, 2, 4, 1, 3, 5).reshape(len(i) * len(j) * len(k), -1)
            out.append((m[i][:, j][:, :, k].flatten(), Kb))
        return out

    def apply_K(self, X, hx, hy):
        """Rows of X times K (from box hx to box hy)."""
        Y = torch.zeros_like(X)
        for idx, Kb in self._K(hx, hy):
            Y[:, idx] = X[:, idx] @ Kb
        return Y

    def B(self):
        Bu = torch.empty((self.npair, self.npair), dtype=torch.float64, device=DEV)
        for s, (gs, hs) in enumerate(zip(self.groups, self.half)):
            for t, (gt, ht) in enumerate(zip(self.groups, self.half)):
                if t < s:
                    continue
                G = self.apply_K(self.F[gs] if len(self.groups) > 1 else self.F, hs, ht)
                Ft = self.F[gt] if len(self.groups) > 1 else self.F
                if len(self.groups) == 1:  # the upper triangle in blocks of rows, mirrored
                    for r in range(0, self.npair, 2048):
                        e = min(self.npair, r + 2048)
                        Bu[r:e, r:] = G[r:e] @ Ft[r:].T
                        Bu[e:, r:e] = Bu[r:e, e:].T
                else:
                    blk = G @ Ft.T
                    Bu[gs[:, None], gt[None, :]] = blk
                    Bu[gt[:, None], gs[None, :]] = blk.T
        i = self.index.flatten()
        return Bu[:, i][i]

    def J(self, D):
        u = D[:, self.mu, self.nu] * torch.where(self.mu == self.nu, 1.0, 2.0).to(torch.float64)
        Ju = self.apply_K(u @ self.F, self.half[0], self.half[0]) @ self.F.T
        return Ju[:, self.index]

    def X(self, Q):
        """Exchange: 2 sum_j X_j K X_j^T with X_j(mu, :) = sum_la q_j(la) F(pair(mu, la), :)."""
        out = torch.zeros((self.nbf, self.nbf), dtype=torch.float64, device=DEV)
        M = self.F[self.index]  # mu, la, m
        for j in range(0, Q.shape[0], 16):
            Xj = torch.einsum("jl,ulm->jum", Q[j:j + 16], M)
            Yj = self.apply_K(Xj.flatten(0, 1), self.half[0], self.half[0]).view_as(Xj)
            out += 2 * torch.einsum("jum,jvm->uv", Yj, Xj)
        return out


def exact(case, seed):
    """What run returns, in 64 bits.  The compressed plan's B is that of the uncompressed one (the dropped singular
    values change it by less than the tensor-core scheme does)."""
    if case["kind"] == "batch":
        return [_Exact(m).J(_densities(seed + i, m.nbf, case["R"])) for i, (_, m) in enumerate(_batch(case, seed))]
    e = _Exact(_molecule(case, seed), tau=1e-20, parts=case.get("parts", 1))
    if case["kind"] == "j":
        return e.J(_densities(seed, e.nbf, case["R"]))
    if case["kind"] == "x":
        return e.X(_orbitals(seed, e.nbf, case["orbs"]))
    return e.B()
