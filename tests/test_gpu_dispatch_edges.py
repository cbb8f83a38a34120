"""Both sides of the rules that choose kernels by size: equal bits where the code claims them, the oracle elsewhere.

Tolerances as in test_gpu_parity.py (relative Frobenius norm): 1e-12 for FP64, 1e-7 for six products.
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


def rel_fro(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", ["split_f16", "split_f16_8", "bf16"])
@pytest.mark.parametrize("natoms", [3, 4, 5])
def test_tile_widths_give_equal_bits(lib, natoms, prec):
    """B_u of 1035 pairs goes in 64-column tiles, of 1830 and 2850 pairs in 128-column ones; its first 128 rows by
    themselves, with tile widths of their own, are the same bits from the diagonal on.  With eight products 128-column
    tiles are two launches (the smaller terms added to C), 64-column ones a single launch."""
    m = synth.workload_spd(1002, natoms=natoms, n=13, P=7)
    pl = lib.Plan(m, prec)
    whole = pl.Bu_rows(0, pl.npair, "factored").cpu().numpy()
    band = pl.Bu_rows(0, 128, "factored").cpu().numpy()
    pl.status()
    assert np.array_equal(np.triu(band), np.triu(whole[:128]))
    pl.close()


def test_eight_products_of_few_and_many_columns_give_equal_bits(lib):
    """J-builds of 64, 100 and 300 densities: one 64-column tile, two, and launches by the waves they take."""
    import torch
    m = synth.workload_spd(1002, natoms=5, n=12, P=6)
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 300), device="cuda")
    pl = lib.Plan(m, "split_f16_8")
    J = pl.jbuild(D)
    for R in (64, 100):
        assert torch.equal(pl.jbuild(D[:R].contiguous()), J[:R])
    pl.status()
    pl.close()


def test_digit_products_of_a_compressed_plan(lib):
    """One class in the natural order: a compressed plan's K has no parity.  Two rows by the CUDA cores beside it."""
    m = synth.workload_spd(1002, natoms=4, cube=8.0, P=20)
    pl = lib.Plan(m, "fp64")
    pl.compress(1e-8)
    lib.lrtei_profile_enable(True)
    lib.lrtei_profile_reset()
    B = pl.assemble_B("factored").cpu().numpy()
    assert lib.lrtei_profile_get("kron")[1] == 0, "the CUDA-core node sum ran: the size does not reach the digit products"
    rows = pl.Bu_rows(5, 7, "factored").cpu().numpy()
    assert lib.lrtei_profile_get("kron")[1] > 0, "two rows took the digit products"
    lib.lrtei_profile_enable(False)
    pl.status()
    pl.close()
    mu, nu = np.triu_indices(m.nbf)
    assert np.array_equal(B, B.T)
    assert rel_fro(B[mu[5:7] * m.nbf + nu[5:7]][:, mu * m.nbf + nu], rows) <= 1e-12


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("split_f16", 1e-7)])
def test_rows_longer_than_shared_memory(lib, prec, tol):
    """Order 31: rows of 29 791 columns are sliced in two passes instead of from shared memory."""
    import torch
    m = synth.workload_spd(1002, natoms=2, cube=4.0, n=31, P=5)
    o = oracle.Oracle.from_molecule(m)
    D = synth.random_densities(5, m.nbf, 32)
    pl = lib.Plan(m, prec)
    B = pl.assemble_B("factored").cpu().numpy()
    J = pl.jbuild(torch.as_tensor(D, device="cuda")).cpu().numpy()
    pl.status()
    pl.close()
    rows = [0, m.nbf + 2, m.nbf ** 2 // 2 + 1, m.nbf ** 2 - 1]
    assert rel_fro(B[rows], o.B_rows(rows)) <= tol
    assert rel_fro(J, o.jbuild_factored(D)) <= tol
