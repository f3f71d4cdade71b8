"""The initial guess at the edges of the gather's row chunks (512) and tiles: its trace and that of its
square, which every stored entry enters, against NumPy, and Gershgorin bounds of one to many rows."""

import numpy as np
import pytest

from synth import dense_from_csr, make_tb_system

pytestmark = pytest.mark.gpu


# FP64 sums of n^2 terms below 1; FP16 hi + lo and TF32 hi + lo operands carry 21 bits or more, BF16 8
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp64e", 1e-13), ("fp16x3", 2.0 ** -20),
                                           ("tf32x3", 2.0 ** -20), ("bf16", 2.0 ** -7)])
@pytest.mark.parametrize("sites", [1, 31, 128, 129, 257])  # 4, 124, 512, 516, 1028 orbitals
def test_initial_guess(precision, tol, sites):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    s = make_tb_system(sites, 1, 3.0, seed=60 + sites)
    plan = gsp2.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                     precision=precision)
    plan.density(torch.from_numpy(s.vals).to("cuda:0"))
    hist = plan.history()
    H = dense_from_csr(s.n, s.rowptr, s.colind, s.vals)
    rad = np.sum(np.abs(H), axis=1) - np.abs(np.diag(H))
    lo, hi = np.min(np.diag(H) - rad), np.max(np.diag(H) + rad)
    assert hist["report"]["eps_min"] == pytest.approx(lo, rel=1e-13, abs=1e-13)
    assert hist["report"]["eps_max"] == pytest.approx(hi, rel=1e-13, abs=1e-13)
    X = (hi * np.eye(s.n) - H) / (hi - lo)
    assert hist["traces"][0] == pytest.approx(np.trace(X), abs=tol * s.n)
    Y = np.sum(X * X)
    want = 2 * np.trace(X) - Y if np.trace(X) <= s.nocc else Y
    assert hist["traces"][1] == pytest.approx(want, abs=tol * s.n)
