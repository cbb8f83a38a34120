"""A staged row whose copy does not arrive in time is reported, as every bounded wait is.

The hook LRTEI_TEST_STALL_STAGED_CYCLES makes the slicing kernels, after their own copy has arrived, wait that long for
a phase of the same barrier that nothing completes.
"""
import os

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


@pytest.mark.parametrize("call", ["rows", "orbitals"])
def test_staged_wait_that_runs_out_reports_timeout_then_recovers(lib, call):
    import torch
    m = synth.workload_small_s()
    pl = lib.Plan(m, "split_f16")
    Q = torch.full((1, m.nbf), 0.25, dtype=torch.float64, device="cuda")
    run = (lambda: pl.Bu_rows(0, pl.npair, "factored")) if call == "rows" else (lambda: pl.exchange(Q))
    ref = run().cpu().numpy()
    pl.status()
    os.environ["LRTEI_TEST_STALL_STAGED_CYCLES"] = "200000"  # ~0.1 ms
    try:
        run()
        torch.cuda.synchronize()
    finally:
        del os.environ["LRTEI_TEST_STALL_STAGED_CYCLES"]
    with pytest.raises(lib.LrteiError) as ei:
        pl.status()
    assert ei.value.status == 4, ei.value
    assert np.array_equal(run().cpu().numpy(), ref)
    pl.status()
    pl.close()
