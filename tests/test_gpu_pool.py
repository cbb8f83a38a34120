"""The library's memory pool gives its memory back with the last plan, but for 2 GiB."""
import pytest

from paper_2210_13069_gb300 import synth

pytestmark = pytest.mark.gpu


def test_pool_keeps_at_most_2_GiB_after_the_last_plan():
    import gc
    import torch
    from paper_2210_13069_gb300 import build_lib, lrtei
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build_lib.build()
    lrtei.load()
    gc.collect()  # plans that other tests left
    torch.cuda.synchronize()
    m = synth.workload_spd()
    small = lrtei.Plan(synth.workload_small_s(), "fp64")
    small.close()  # modules and the like are loaded now
    nb2 = m.nbf ** 2
    B = torch.empty((nb2, nb2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pl = lrtei.Plan(m, "split_f16")
    free0 = torch.cuda.mem_get_info()[0]
    pl.assemble_B(out=B)
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held > 3 << 30, "the case is too small to show anything"
    pl.close()
    torch.cuda.synchronize()
    left = free0 - torch.cuda.mem_get_info()[0]
    assert left <= (2 << 30) + (64 << 20), f"{left / 2**30:.2f} GiB kept"
