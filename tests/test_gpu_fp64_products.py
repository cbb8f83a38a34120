"""FP64 J-builds at the edges of their kernels, against the oracle's factored J-build.

Orders of one, odd and even (the Chebyshev coefficients' parity classes), densities from one row to more than one
group of eight (the per-thread groups and the two forms of the node sum), a box that is not a cube.  Tolerance: the
1e-12 of the FP64 path (relative Frobenius norm), as in test_gpu_parity.py.
"""
import numpy as np
import pytest

import oracle
from paper_2210_13069_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    from paper_2210_13069_gb300 import build_lib, lrtei
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build_lib.build()
    lrtei.load()
    return lrtei


def molecule(n, P, natoms=2, box=False):
    m = synth.random_molecule(4101, natoms=natoms, cube=4.0, nprim=2, alpha_range=(0.15, 40.0), omega=0.45, n=n, P=P)
    if box:
        m.box_lo, m.box_hi = np.array([-4.0, -3.5, -5.0]), np.array([8.0, 7.5, 6.0])
    return m


def rel_fro(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,P,R,box", [(1, 1, 1, False), (2, 3, 2, False), (7, 9, 3, True), (16, 5, 4, False),
                                       (9, 33, 5, False), (12, 8, 8, True), (13, 6, 19, False)])
def test_jbuild_fp64_orders_and_counts(lib, n, P, R, box):
    import torch
    m = molecule(n, P, box=box)
    D = synth.random_densities(5, m.nbf, R)
    ref = oracle.Oracle.from_molecule(m).jbuild_factored(D)
    pl = lib.Plan(m, "fp64")
    Dd = torch.as_tensor(D, device="cuda")
    J = pl.jbuild(Dd)
    J2 = pl.jbuild(Dd, out=torch.empty_like(J)).cpu().numpy()
    pl.status()
    J = J.cpu().numpy()
    assert rel_fro(J, ref) <= 1e-12
    assert np.array_equal(J, J2) and np.array_equal(J, J.transpose(0, 2, 1))
    pl.close()


def test_jbuild_fp64_nonfinite_density_is_reported(lib):
    import torch
    m = molecule(6, 5)
    D = synth.random_densities(5, m.nbf, 3)
    D[1, 0, 0] = np.inf
    pl = lib.Plan(m, "fp64")
    J = pl.jbuild(torch.as_tensor(D, device="cuda")).cpu().numpy()
    with pytest.raises(lib.LrteiError) as ei:
        pl.status()
    assert ei.value.status == 5
    ref = oracle.Oracle.from_molecule(m).jbuild_factored(D[[0, 2]])
    assert rel_fro(J[[0, 2]], ref) <= 1e-12 and not np.isfinite(J[1]).any()
    pl.close()


# The FP64 path on the tensor cores (digit products).  Sizes that reach it: ragged last tiles of the pairs (120 and
# 465 pairs against 128-row tiles), orders whose classes fill and miss 64 columns, one to three 32-column density tiles.
@pytest.mark.parametrize("n,P,natoms", [(24, 32, 2), (21, 40, 3), (17, 24, 4)])
def test_B_fp64_digit_products_against_oracle_rows(lib, n, P, natoms):
    m = molecule(n, P, natoms=natoms)
    o = oracle.Oracle.from_molecule(m)
    pl = lib.Plan(m, "fp64")
    lib.lrtei_profile_enable(True)
    lib.lrtei_profile_reset()
    B = pl.assemble_B("factored")
    assert lib.lrtei_profile_get("kron")[1] == 0, "the CUDA-core node sum ran: the size does not reach the digit products"
    lib.lrtei_profile_enable(False)
    pl.status()
    nb2 = m.nbf ** 2
    rows = [0, m.nbf + 2, nb2 // 2 + 1, nb2 - 1]
    B = B.cpu().numpy()
    assert np.array_equal(B, B.T)
    assert rel_fro(B[rows], o.B_rows(rows)) <= 1e-12
    # a band that starts and ends inside 128-row tiles (B row of the unique pair (0, nu) is nu)
    r0, r1 = 13, min(pl.npair - 3, 400)
    band = pl.Bu_rows(r0, r1, "factored").cpu().numpy()
    cols = [ka * m.nbf + la for ka in range(m.nbf) for la in range(ka, m.nbf)]
    assert rel_fro(band[:m.nbf - r0], B[r0:m.nbf][:, cols]) <= 1e-13
    assert rel_fro(band, B[cols[r0:r1]][:, cols]) <= 1e-13
    pl.close()


@pytest.mark.parametrize("R", [6, 31, 32, 33, 70])
def test_jbuild_fp64_digit_products(lib, R):
    import torch
    m = molecule(19, 21, natoms=4)
    D = synth.random_densities(6, m.nbf, R)
    pl = lib.Plan(m, "fp64")
    Dd = torch.as_tensor(D, device="cuda")
    lib.lrtei_profile_enable(True)
    lib.lrtei_profile_reset()
    J = pl.jbuild(Dd).cpu().numpy()
    assert lib.lrtei_profile_get("kron")[1] == 0
    lib.lrtei_profile_enable(False)
    pl.status()
    assert rel_fro(J, oracle.Oracle.from_molecule(m).jbuild_factored(D)) <= 1e-12
    D[1, 2, 3] = D[1, 3, 2] = np.nan  # a density that is not a number spoils its own J only, and is reported
    Jn = pl.jbuild(torch.as_tensor(D, device="cuda")).cpu().numpy()
    with pytest.raises(lib.LrteiError) as ei:
        pl.status()
    assert ei.value.status == 5
    assert np.isnan(Jn[1]).all() and np.array_equal(Jn[0], J[0]) and np.array_equal(Jn[2:], J[2:])
    pl.close()
