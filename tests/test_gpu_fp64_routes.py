"""FP64 calls give the same bits whatever was called on the plan before (the digit operands of one call do not draw
another call to the digit route)."""
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


def test_rows_before_and_after_a_jbuild(lib):
    """24 rows of B_u at order 24: cheaper on the CUDA cores with K still to build, in digits without."""
    import torch
    m = synth.workload_spd(1002, natoms=2, cube=4.0)
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 8), device="cuda")
    pl = lib.Plan(m, "fp64")
    first = pl.Bu_rows(0, 24, "factored")
    J = pl.jbuild(D)
    B = pl.assemble_B("factored")
    assert torch.equal(pl.Bu_rows(0, 24, "factored"), first)
    fresh = lib.Plan(m, "fp64")
    assert torch.equal(fresh.assemble_B("factored"), B)
    assert torch.equal(fresh.jbuild(D), J)
    pl.status()
    pl.close()
    fresh.close()


def test_jbuild_of_high_order_before_and_after_B(lib):
    """Order 33: a J-build does not build K, but B does."""
    import torch
    m = synth.workload_spd(1002, natoms=4, cube=8.0, n=33, P=16)
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 8), device="cuda")
    pl = lib.Plan(m, "fp64")
    J = pl.jbuild(D)
    pl.assemble_B("factored")
    assert torch.equal(pl.jbuild(D, out=torch.empty_like(D)), J)
    pl.status()
    pl.close()
