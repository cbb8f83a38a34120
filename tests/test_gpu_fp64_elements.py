"""FP64 B and J-builds element by element on the tensor-core (digit product) route.

A norm does not see the small elements of B, which FP64 sums of products hold to a few units of 2^-53 of the sum of
their terms' magnitudes.  The reference is formed in extended precision from the plan's own moments, coefficients and
weights, and each element has to lie within that model:

    |B - ref| <= c 2^-53 (|F| |K| |F|^T),  c = 2 (I + 3) + (P + 4) + 2 sqrt(n^3):

the roundings of the I terms of F_u on both sides, those of the P terms of K, and a random walk over the two
contractions of length n^3.  J of a density with one nonzero pair is a row of B.
"""
import numpy as np
import pytest

from paper_2210_13069_gb300 import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def lib():
    import torch
    from paper_2210_13069_gb300 import build_lib, lrtei
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build_lib.build()
    lrtei.load()
    return lrtei


def kron(A, w, X):
    """sum_p w_p (A_x^p (x) A_y^p (x) A_z^p) on the rows of X."""
    P, n = A.shape[1], A.shape[2]
    X = X.reshape(-1, n, n, n)
    Y = np.zeros_like(X)
    for p in range(P):
        t = np.tensordot(X, A[2, p], (3, 1))
        t = np.tensordot(t, A[1, p], (2, 1))
        t = np.tensordot(t, A[0, p], (1, 1))
        Y += w[p] * t.transpose(0, 3, 2, 1)
    return Y.reshape(len(Y), -1)


@pytest.mark.parametrize("seed,n,P,omega", [(1, 16, 20, 0.4), (4101, 13, 17, 0.45)])
def test_small_elements_have_fp64_accuracy(lib, seed, n, P, omega):
    import torch
    m = synth.workload_spd(seed, natoms=2, cube=4.0, omega=omega, n=n, P=P)
    pl = lib.Plan(m, "fp64")
    npair, I = pl.npair, pl.info["nrows"] // pl.npair
    S, C, _, w, c = (x.cpu().numpy() for x in pl.factors())
    pref = LD(m.omega) / np.sqrt(LD(np.pi))
    rows = np.random.default_rng(seed).choice(npair, 12, replace=False)

    def F_of(S, c, dt):
        S = S.reshape(3, npair, I, n)
        yz = (S[1][..., :, None].astype(dt) * S[2][..., None, :].astype(dt)).reshape(npair, I, n * n)
        x = S[0].astype(dt) * c.reshape(npair, I, 1).astype(dt)
        return np.stack([sum(x[r, j][:, None] * yz[r, j][None, :] for j in range(I)).ravel() for r in range(npair)])

    F, A = F_of(S, c, LD), C.reshape(3, P, n, n).astype(LD)
    ref = pref * (kron(A, w.astype(LD), F[rows]) @ F.T)
    Fa = F_of(np.abs(S), np.abs(c), np.float64)
    size = float(pref) * (kron(np.abs(C.reshape(3, P, n, n)), np.abs(w), Fa[rows]) @ Fa.T)
    bound = (2 * (I + 3) + (P + 4) + 2 * n ** 1.5) * 2.0 ** -53 * size

    lib.lrtei_profile_enable(True)
    lib.lrtei_profile_reset()
    B = pl.assemble_B("factored").cpu().numpy()
    mu, nu = np.triu_indices(m.nbf)
    D = torch.zeros((32, m.nbf, m.nbf), dtype=torch.float64, device="cuda")
    for q, r in enumerate(rows):
        D[q, mu[r], nu[r]] = D[q, nu[r], mu[r]] = 1.0 if mu[r] == nu[r] else 0.5
    J = pl.jbuild(D).cpu().numpy()
    assert lib.lrtei_profile_get("kron")[1] == 0, "the CUDA-core node sum ran: the size does not reach the digit products"
    lib.lrtei_profile_enable(False)
    pl.status()
    pl.close()
    Bu = B[mu[rows] * m.nbf + nu[rows]][:, mu * m.nbf + nu]
    for got in (Bu, J[:len(rows), mu, nu]):
        err = np.abs(got.astype(LD) - ref).astype(np.float64)
        print(f"seed {seed}: largest error {np.max(err / np.maximum(bound, 1e-300)):.3f} of the bound")
        assert (err <= bound).all()
