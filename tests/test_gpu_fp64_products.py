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
