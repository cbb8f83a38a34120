"""Split-precision B and J-builds at the edges of the tensor-core products, against the oracle.

Orders whose 16-deep K blocks hold one, several or all parity classes (n = 1, 5, 8, 13, 16, 21), pair counts around
128-row tiles, densities around the 32-, 64- and 128-column tiles, bands of rows that start inside a tile.  Tolerances
as in test_gpu_parity.py (relative Frobenius norm): 1e-7 for six and eight products, 5e-3 for plain BF16 (one rounding
of 2^-9 per element and a cancellation of ~150 leave about 1e-3).
"""
import numpy as np
import pytest

import oracle
from paper_2210_13069_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = {"split_f16": 1e-7, "split_f16_8": 1e-7, "bf16": 5e-3}


@pytest.fixture(scope="module")
def lib():
    import torch
    from paper_2210_13069_gb300 import build_lib, lrtei
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build_lib.build()
    lrtei.load()
    return lrtei


def molecule(n, P, natoms=2):
    return synth.random_molecule(4201, natoms=natoms, cube=4.0, nprim=2, alpha_range=(0.15, 40.0), omega=0.45, n=n, P=P)


def rel_fro(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", ["split_f16", "split_f16_8", "bf16"])
@pytest.mark.parametrize("n,P,natoms", [(1, 2, 1), (5, 4, 1), (8, 6, 2), (13, 7, 2), (16, 5, 1), (21, 6, 2)])
def test_B_orders_and_ragged_tiles(lib, prec, n, P, natoms):
    m = molecule(n, P, natoms)
    o = oracle.Oracle.from_molecule(m)
    pl = lib.Plan(m, prec)
    B = pl.assemble_B("factored").cpu().numpy()
    pl.status()
    rows = [0, m.nbf + 1, m.nbf ** 2 - 1] if natoms > 1 else list(range(m.nbf ** 2))
    assert np.array_equal(B, B.T)
    assert rel_fro(B[rows], o.B_rows(rows)) <= TOL[prec]
    r0, r1 = 5, min(pl.npair, 140)
    band = pl.Bu_rows(r0, r1, "factored").cpu().numpy()
    cols = [ka * m.nbf + la for ka in range(m.nbf) for la in range(ka, m.nbf)]
    # the triangle's rows and a band's rows contract in the two orders of the product: rounding only
    assert rel_fro(band, B[cols[r0:r1]][:, cols]) <= 2 * TOL[prec]
    pl.close()


@pytest.mark.parametrize("prec", ["split_f16", "split_f16_8"])
@pytest.mark.parametrize("R", [1, 33, 64, 65, 130])
def test_jbuild_density_tiles(lib, prec, R):
    import torch
    m = molecule(11, 6)
    D = synth.random_densities(7, m.nbf, R)
    pl = lib.Plan(m, prec)
    J = pl.jbuild(torch.as_tensor(D, device="cuda")).cpu().numpy()
    pl.status()
    assert rel_fro(J, oracle.Oracle.from_molecule(m).jbuild_factored(D)) <= TOL[prec]
    pl.close()


# n^3 a multiple of eight (orbital rows sliced in place) and not (through the permuted copy); one orbital and several.
@pytest.mark.parametrize("prec", ["split_f16", "split_f16_8"])
@pytest.mark.parametrize("n,orbs", [(9, 3), (10, 1), (12, 5)])
def test_exchange_operand_layouts(lib, prec, n, orbs):
    import torch
    m = molecule(n, 5)
    Q = np.random.Generator(np.random.Philox(11)).normal(0.0, 1.0 / np.sqrt(m.nbf), size=(orbs, m.nbf))
    B = oracle.Oracle.from_molecule(m).assemble_B().reshape(m.nbf, m.nbf, m.nbf, m.nbf)
    ref = 2.0 * np.einsum("jl,jk,mlkn->mn", Q, Q, B, optimize=True)
    pl = lib.Plan(m, prec)
    K = pl.exchange(torch.as_tensor(Q, device="cuda")).cpu().numpy()
    pl.status()
    assert rel_fro(K, ref) <= TOL[prec]
    pl.close()


# 32-, 64- and 128-column tiles of orbitals, against the FP64 plan of the same molecule.
@pytest.mark.parametrize("prec", ["split_f16", "split_f16_8"])
@pytest.mark.parametrize("orbs", [32, 33, 65])
def test_exchange_orbital_tiles(lib, prec, orbs):
    import torch
    m = molecule(8, 4, 5)
    Q = torch.as_tensor(np.random.Generator(np.random.Philox(12)).normal(0.0, 1.0 / np.sqrt(m.nbf), size=(orbs, m.nbf)),
                        device="cuda")
    K = []
    for p in ("fp64", prec):
        pl = lib.Plan(m, p)
        K.append(pl.exchange(Q).cpu().numpy())
        pl.status()
        pl.close()
    assert rel_fro(K[1], K[0]) <= TOL[prec]
