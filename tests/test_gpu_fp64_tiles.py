"""Native FP64 steps on 16 x 16 tiles: P and the adjoint against the oracle at sizes around a
tile, and the idempotency report against the oracle's residual."""

import numpy as np
import pytest

import oracle
from synth import dense_from_csr, make_tb_system, random_symmetric_on_pattern

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites,parts", [(1, 1), (4, 1), (5, 1), (9, 3), (33, 2)])  # 4, 16, 20, 36, 132 orbitals
def test_native_fp64_at_tile_edges(sites, parts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    s = make_tb_system(sites, parts, 3.0, seed=40 + sites)
    plan = gsp2.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                     ckpt_every=3, report_idem=1)
    p = plan.density(torch.from_numpy(s.vals).to("cuda:0"))
    hist = plan.history()
    ref = oracle.gsp2(s.n, s.rowptr, s.colind, s.vals, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind,
                      alphas=hist["alphas"])
    assert np.max(np.abs(p.cpu().numpy() - ref.p_on_pattern(plan.p_colptr, plan.p_rowind))) <= 1e-10
    res = sum(np.sum((X @ X - X)[:, :c] ** 2) for X, c in zip(ref.X, ref.ncore))
    assert hist["report"]["idem_fro"] == pytest.approx(np.sqrt(res / s.n), rel=1e-6, abs=1e-12)
    A = dense_from_csr(s.n, s.rowptr, s.colind, random_symmetric_on_pattern(s.rowptr, s.colind, 5678))
    cols = np.repeat(np.arange(s.n), np.diff(plan.p_colptr))
    pb = A[plan.p_rowind, cols]
    Pbar = np.zeros((s.n, s.n))
    Pbar[plan.p_rowind, cols] = pb
    got = plan.backward(torch.from_numpy(pb).to("cuda:0")).cpu().numpy()
    want = oracle.gsp2_adjoint(s.n, s.rowptr, s.colind, s.vals, ref, Pbar)
    assert np.max(np.abs(got - want)) <= 1e-9 * max(1.0, np.max(np.abs(want)))
