"""Stream captures beside and around the library's calls.

A plan that gives buffers back in one thread (compression, the FP64 F_u of a J-build) leaves another thread's capture
alone (captures of the thread-local kind, as the library's own of its J-builds are).
"""
import threading

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


def molecule():
    return synth.random_molecule(4301, natoms=2, cube=4.0, nprim=1, alpha_range=(0.15, 40.0), omega=0.45, n=8, P=6)


@pytest.mark.parametrize("what", ["jbuild", "compress"])
def test_plans_of_another_thread_leave_a_capture_alone(lib, what):
    import torch
    m = molecule()
    x = torch.zeros(1000, device="cuda")
    pl = lib.Plan(m, "split_f16")
    ref = pl.assemble_B("factored")
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 2), device="cuda")
    J = torch.empty_like(D)
    errors = []

    def other():
        try:
            if what == "compress":
                pl.compress(0.0)  # full rank: releases the operands, B is the same
            else:
                pl.jbuild(D, out=J)  # F_u is sliced twice then, its FP64 copy goes
        except Exception as e:  # reported below, in the test's thread
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=side, capture_error_mode="thread_local"):
        x += 1.0
        t = threading.Thread(target=other)
        t.start()
        t.join()
        x += 1.0
    assert not errors, errors
    g.replay()
    torch.cuda.synchronize()
    assert (x == 2.0).all()
    if what == "compress":
        B = pl.assemble_B("factored")
        assert torch.linalg.norm(B - ref) <= 1e-7 * torch.linalg.norm(ref)
    else:
        K = torch.einsum("rc,qc->qr", ref, D.reshape(2, -1)).reshape(D.shape)
        assert torch.linalg.norm(J - K) <= 1e-7 * torch.linalg.norm(K)
    pl.close()


CALLS = {
    "B split factored": ("split_f16", lambda pl, D, Q: pl.assemble_B("factored")),
    "B split Hadamard": ("split_f16", lambda pl, D, Q: pl.assemble_B("hadamard")),
    "B fp64 factored": ("fp64", lambda pl, D, Q: pl.assemble_B("factored")),
    "B fp64 Hadamard": ("fp64", lambda pl, D, Q: pl.assemble_B("hadamard")),
    "B fp32": ("fp32", lambda pl, D, Q: pl.assemble_B("factored")),
    "J split": ("split_f16_8", lambda pl, D, Q: pl.jbuild(D)),
    "J fp64": ("fp64", lambda pl, D, Q: pl.jbuild(D)),
    "K split": ("split_f16", lambda pl, D, Q: pl.exchange(Q)),
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_operands_of_a_captured_first_call_exist_before_the_replay(lib, name):
    """The first call of a plan inside a relaxed capture: its operands are there for plain calls, replayed or not."""
    import torch
    prec, call = CALLS[name]
    m = molecule()
    D = torch.as_tensor(synth.random_densities(5, m.nbf, 3), device="cuda")
    Q = torch.as_tensor(np.random.default_rng(3).normal(size=(2, m.nbf)), device="cuda")
    fresh = lib.Plan(m, prec)
    ref = call(fresh, D, Q)
    pl = lib.Plan(m, prec)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="relaxed"):
        out = call(pl, D, Q)
    assert torch.equal(call(pl, D, Q), ref)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    pl.status()
    del g
    pl.close()
    fresh.close()


@pytest.mark.parametrize("mode", ["global", "thread_local"])
def test_a_B_that_asks_for_the_free_memory_can_be_captured(lib, mode):
    """105 functions of order 18 in digit products: 1.6 GB of scratch, which the call looks for."""
    import torch
    m = synth.workload_spd(1002, natoms=7, n=18, P=20)
    pl = lib.Plan(m, "fp64")
    ref = pl.assemble_B("factored")
    out = torch.empty_like(ref)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode=mode):
        pl.assemble_B("factored", out=out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    del g
    pl.close()
