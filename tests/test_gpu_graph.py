"""The dependency graph built on the device (gsp2_threshold_graph) against the construction on the
host from the stored values of P: thresholds from none to all entries, sizes around the bitmap's
words and the block, uneven and single-vertex parts, one part, NaN in P."""

import numpy as np
import pytest

from synth import make_tb_system, make_workload
from synth.tb import core_weights

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


def host_graph(plan, pv, tau):
    n = plan.n
    cols = np.repeat(np.arange(n), np.diff(plan.p_colptr))
    keep = (np.abs(pv) > tau) & (plan.p_rowind != cols)
    r, c = plan.p_rowind[keep].astype(np.int64), cols[keep]
    pairs = np.unique(np.concatenate([r, c, np.arange(n)]) * n + np.concatenate([c, r, np.arange(n)]))
    return np.searchsorted(pairs // n, np.arange(n + 1)), (pairs % n).astype(np.int32)


CASES = {
    "one32": lambda: make_tb_system(8, 1, 3.0, seed=3),        # 32 vertices: one word
    "single": lambda: make_tb_system(9, 9, 3.0, seed=4),       # one site per part, 36 vertices
    "ragged1044": lambda: make_tb_system(261, 7, 3.3, seed=5),
    "uneven2400": lambda: make_tb_system(600, 24, 4.0, seed=6, weights=core_weights(24, 7, 4.0, 76.0)),
    "tb4k": lambda: make_workload("tb4k"),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_graph_matches_the_host_construction(g, case):
    import torch
    s = CASES[case]()
    plan = g.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                  ckpt_every=0, bind=True)
    rng = np.random.default_rng(s.n)
    # values over many magnitudes, not symmetric between the two stored orders, some NaN
    pv = rng.standard_normal(plan.nnz_p) * 10.0 ** rng.uniform(-8, 0, plan.nnz_p)
    pv[rng.integers(0, plan.nnz_p, 5)] = np.nan
    p = torch.from_numpy(pv).to("cuda:0")
    for tau in (0.0, 1e-6, 1e-2, 1e9):
        rp, ci = plan.threshold_graph(p, tau)
        want_rp, want_ci = host_graph(plan, pv, tau)
        np.testing.assert_array_equal(rp, want_rp)
        np.testing.assert_array_equal(ci, want_ci)
