"""Calls on a nearly full device: what a route allocates beyond its operands is part of the decision to take it.

A tensor fills the device but for what the case names.  Each call has to end well where a route of less scratch exists.
"""
import contextlib

import numpy as np
import pytest

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


@contextlib.contextmanager
def leave_free(nbytes):
    """Leaves nbytes of the device's memory free for a while."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    assert free > nbytes, "the device is not free enough for this case"
    filler = torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del filler
        torch.cuda.empty_cache()


def rel_fro(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("natoms,n,free", [(21, 24, 109_500_000_000), (15, 18, 21_000_000_000)])
def test_fp64_B_where_the_split_partials_do_not_fit(lib, natoms, n, free):
    """49 770 pairs of order 24: K of 216 pieces goes in three splits, 59 GB of partial sums beside the 53 GB of the
    operands and B_u; 25 425 pairs of order 18: two splits, 10 beside 12 GB.  B has to come in bands of digit products
    (1e-12 as in test_gpu_fp64_products.py)."""
    import torch
    m = synth.workload_spd(1002, natoms=natoms, n=n, P=20)
    pl = lib.Plan(m, "fp64")
    nb2 = m.nbf ** 2
    B = torch.empty((nb2, nb2), dtype=torch.float64, device="cuda")
    lib.lrtei_profile_enable(True)
    lib.lrtei_profile_reset()
    with leave_free(free):
        pl.assemble_B("factored", out=B)
    assert lib.lrtei_profile_get("kron")[1] == 0, "the CUDA-core route ran"
    lib.lrtei_profile_enable(False)
    pl.status()
    r0 = 7
    ref = pl.Bu_rows(r0, r0 + 2, "factored").cpu().numpy()  # two rows: the CUDA-core route
    mu, nu = np.triu_indices(m.nbf)
    cols = torch.as_tensor(mu * m.nbf + nu, device="cuda")
    for i in range(2):
        row = B[mu[r0 + i] * m.nbf + nu[r0 + i]][cols].cpu().numpy()
        assert rel_fro(row, ref[i]) <= 1e-12
    pl.close()


@pytest.mark.parametrize("precision,R,free", [("fp32", 8192, 3_000_000_000), ("fp64", 16384, 2_900_000_000)])
def test_jbuild_of_many_densities_has_bounded_scratch(lib, precision, R, free):
    """60 functions of order 16.  FP32 plans (CUDA cores, 38 partial sums of X) would take 10 GB for all densities at
    once, FP64 ones (digits and their vectors) 6.6 GB."""
    import torch
    import oracle
    m = synth.workload_spd(1002, natoms=4, cube=8.0, n=16, P=20)
    pl = lib.Plan(m, precision)
    few = torch.as_tensor(synth.random_densities(5, m.nbf, 7), device="cuda")
    D = few[torch.arange(R, device="cuda") % 7].contiguous()
    J = torch.empty_like(D)
    with leave_free(free):
        pl.jbuild(D, out=J)
    pl.status()
    ref = oracle.Oracle.from_molecule(m).jbuild_factored(few.cpu().numpy())
    for q in (0, 31, 1023, R // 2 + 3, R - 1):
        assert rel_fro(J[q].cpu().numpy(), ref[q % 7]) <= 1e-12
    pl.close()


def test_adaptive_B_where_the_blocks_of_all_pairs_do_not_fit(lib):
    """150 functions in eight boxes of about 1400 pairs, order 13: G, its slices and the blocks of all 36 pairs of boxes
    take 2.5 GB beside B_u (1.0 GB) and F_u (0.4 GB); one after the other 0.1."""
    import torch
    m = synth.workload_spd(1002, natoms=10, n=13, P=11)
    pl = lib.Plan(m, "split_f16", adaptive=(1e-20, 8))
    nb2 = m.nbf ** 2
    B = torch.empty((nb2, nb2), dtype=torch.float64, device="cuda")
    with leave_free(3_000_000_000):
        pl.assemble_B(out=B)
    pl.status()
    tight = B.clone()
    pl.assemble_B(out=B)
    pl.status()
    assert torch.equal(B, tight)  # the same products, tile by tile
    pl.close()


def test_the_idle_pool_counts_as_free_memory(lib):
    """150 functions of order 18: a B in digit products needs 4.8 GB of scratch and leaves about 3.9 in the pool.  With
    5 GB free beside that it is formed whole again, not in bands."""
    import torch
    m = synth.workload_spd(1002, natoms=10, n=18, P=20)
    pl = lib.Plan(m, "fp64")
    nb2 = m.nbf ** 2
    B = torch.empty((nb2, nb2), dtype=torch.float64, device="cuda")
    pl.assemble_B("factored", out=B)  # its operands are built
    first = B.clone()
    with leave_free(5_000_000_000):
        lib.lrtei_profile_enable(True)
        lib.lrtei_profile_reset()
        pl.assemble_B("factored", out=B)
        products = lib.lrtei_profile_get("gemm_fp64")[1]
        lib.lrtei_profile_enable(False)
    pl.status()
    assert products == 2, "G and B_u: the rows came in bands"
    assert torch.equal(B, first)
    pl.close()


@pytest.mark.parametrize("batched", [False, True])
def test_many_fp64_plans_share_the_device(lib, batched):
    """Sixty plans of 180 functions: 108 GB of F_u in FP64, which fit, and 430 GB as digit operands, which do not."""
    import torch
    m = synth.workload_spd()
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 4), device="cuda")
    plans = [lib.Plan(m, "fp64") for _ in range(60)]
    J = [torch.empty_like(D) for _ in plans]
    if batched:
        lib.lrtei_jbuild_batched([p.plan for p in plans], [D] * 60, [4] * 60, J)
    else:
        for p, j in zip(plans, J):
            p.jbuild(D, out=j)
    torch.cuda.synchronize()
    for p in (plans[0], plans[59]):
        p.status()
    a, b = J[0].cpu().numpy(), J[59].cpu().numpy()  # digit products, CUDA cores
    assert rel_fro(a, b) <= 1e-12
    for p in plans:
        p.close()
