"""Emulated FP64 steps in wide K slices (plans of more than 3 tiles per SM whose parts average 512
orbitals or more): P and the adjoint against the native FP64 path on the same branches, for ragged
parts, whole and in K halves, and for one part whose K takes two rounds."""

import numpy as np
import pytest

from synth import make_tb_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites,parts,radius,split", [(900, 28, 5.0, -1), (900, 28, 5.0, 1), (975, 1, 3.0, -1)])
def test_wide_slices(sites, parts, radius, split):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    s = make_tb_system(sites, parts, radius, seed=70 + parts)
    h = torch.from_numpy(s.vals).to("cuda:0")
    out = {}
    alpha = None
    for prec in ("fp64e", "fp64"):
        plan = gsp2.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                         ckpt_every=4, precision=prec, split_k=split if prec == "fp64e" else -1)
        blocks = [-(-int(z) // 128) for z in plan.part_sizes]
        assert sum(b * (b + 1) // 2 for b in blocks) > 3 * 152
        if alpha is None:
            p = plan.density(h)
            hist = plan.history()
            alpha = torch.zeros(plan.alpha_len, dtype=torch.int8, device="cuda:0")
            alpha[:len(hist["alphas"])] = torch.tensor(hist["alphas"], dtype=torch.int8)
            torch.manual_seed(3)
            pb = torch.randn(plan.nnz_p, dtype=torch.float64, device="cuda:0")
        else:
            p = plan.density(h, alpha=alpha, mode="replay", nsteps=len(hist["alphas"]))
        out[prec] = (p.cpu().numpy(), plan.backward(pb).cpu().numpy())
        del plan
    assert np.max(np.abs(out["fp64e"][0] - out["fp64"][0])) <= 1e-10
    want = out["fp64"][1]
    assert np.max(np.abs(out["fp64e"][1] - want)) <= 1e-9 * max(1.0, np.max(np.abs(want)))
