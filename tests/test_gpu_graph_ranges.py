"""gsp2_threshold_graph beyond one pass: more columns than its buffer holds (the rows then come in ranges)
and more vertices than a bitmap of shared memory holds (windows of 1,572,864)."""

import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    return gsp2


def check(rp, ci, rows, cols, n):
    """The CSR graph (rp, ci) is that of the edges (rows, cols), both ways, and the diagonal."""
    key = np.concatenate([rows * n + cols, cols * n + rows, np.arange(n) * (n + 1)])
    key.sort()
    key = key[np.concatenate([[True], key[1:] != key[:-1]])]
    assert rp[0] == 0 and rp[n] == len(key)
    np.testing.assert_array_equal(np.diff(rp), np.bincount(key // n, minlength=n))
    np.testing.assert_array_equal(ci, key % n)


def test_rows_in_two_ranges(g):
    import torch
    s = make_workload("tb30k")
    plan = g.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                  ckpt_every=0, bind=True)
    p = torch.rand(plan.nnz_p, dtype=torch.float64, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(9))
    tau = 0.2
    rp, ci = plan.threshold_graph(p, tau)
    assert len(ci) > 16 << 20  # columns of the buffer
    keep = p.cpu().numpy() > tau
    cols = np.repeat(np.arange(s.n), np.diff(plan.p_colptr))[keep]
    check(rp, ci, plan.p_rowind[keep].astype(np.int64), cols, s.n)


def test_vertices_beyond_one_window(g):
    import torch
    n, size = 1_600_000, 128  # chains of 128 orbitals, each a part
    part = (np.arange(n) // size).astype(np.int32)
    rowptr = np.arange(n + 1, dtype=np.int64)
    none = np.zeros(n + 1, np.int64)
    plan = g.GSP2(n, rowptr, np.arange(n, dtype=np.int32), n // 2, part, n // size, none, np.zeros(0, np.int32),
                  device="cuda:0", ckpt_every=0, bind=True)
    p = torch.rand(plan.nnz_p, dtype=torch.float64, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(3))
    tau = 0.995
    rp, ci = plan.threshold_graph(p, tau)
    at = torch.nonzero(p > tau)[:, 0].cpu().numpy()
    cols = np.searchsorted(plan.p_colptr, at, side="right") - 1
    check(rp, ci, plan.p_rowind[at].astype(np.int64), cols, n)
