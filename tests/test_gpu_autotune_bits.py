"""The autotuner's choice never changes the results of an emulated FP64 plan: split-K work items are
candidates only where the plan's split and whole items round at the same K."""

import numpy as np
import pytest

from synth import make_workload
from synth.tb import make_tb_system

pytestmark = pytest.mark.gpu

CASES = {
    "tb512": lambda: make_workload("tb512"),            # 24 tiles: splits by default
    "tiles48": lambda: make_tb_system(300, 12, 3.0, seed=8),  # a few more than a quarter of the SMs
    "tb4k": lambda: make_workload("tb4k"),              # 193 tiles: whole items
}


@pytest.mark.parametrize("case,split", [("tb512", -1), ("tb512", 0), ("tiles48", -1), ("tb4k", -1), ("tb4k", 1)])
def test_autotuned_plan_gives_the_same_bits(case, split):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    s = CASES[case]()
    plan = gsp2.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                     precision="fp64e", ckpt_every=0, split_k=split)
    h = torch.from_numpy(s.vals).to("cuda:0")
    p0 = plan.density(h).cpu().numpy()
    split0 = plan.info.split_k
    blocks = [-(-int(z) // 128) for z in plan.part_sizes]
    tiles = sum(b * (b + 1) // 2 for b in blocks)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if split < 0 and min(plan.part_sizes) > 128:
        assert split0 == (1 if tiles <= sms // 4 else 0), tiles
    rep = plan.autotune(h, trials=1)
    assert np.array_equal(p0, plan.density(h).cpu().numpy())
    if split < 0 and split0 == 0:  # whole items by default round at other K than split ones
        assert all(c["split_k"] == 0 for c in rep["candidates"])
