"""The five FP16 digits of the emulated FP64 step and the fifteen products it keeps.

On the CPU, from their definition and independently of the kernels: the digits reconstruct x
to 2^-50 and are exact in FP16 at the scales they are stored with, also for |x| up to 2; the
accumulators that must be exact stay below 2^24 on dense rows at K = 2048; the products left
out are smaller than what seven 7-bit digits leave out.  On the GPU: one step against the
FP64 product at the sizes where the kernel changes shape."""

import numpy as np
import pytest

WIDTHS = (11, 8, 11, 8, 11)
E = np.cumsum(WIDTHS)
RHO = (-3, -4, -2, -3, -1)


def digits(X):
    """S_0 .. S_4 with round(x 2^49) = sum_t S_t 2^(49 - e_t): balanced for t >= 1, S_0 the
    rest, kept even beyond 2^11 (S_1 takes the odd unit)."""
    r = np.rint(np.asarray(X, np.longdouble) * np.longdouble(2) ** int(E[-1])).astype(np.int64)
    S = [None] * 5
    for t in range(4, 0, -1):
        b = 1 << WIDTHS[t]
        S[t] = ((r + b // 2) % b) - b // 2
        r = (r - S[t]) // b
    odd = np.where(np.abs(r) > 2048, r & 1, 0)
    S[0], S[1] = r - odd, S[1] + 256 * odd
    return S


def test_digits_are_exact_in_fp16():
    rng = np.random.default_rng(5)
    x = np.concatenate([rng.uniform(-1, 1, 20000), rng.uniform(-1.99, 1.99, 2000), [0, 1, -1, 1 + 2.0 ** -12, 2.0 ** -50]])
    S = digits(x)
    w = sum(S[t] * (1 << int(E[-1] - E[t])) for t in range(5))
    assert np.array_equal(w, np.rint(x.astype(np.longdouble) * np.longdouble(2) ** 49).astype(np.int64))
    for t in range(5):
        f = S[t] * 2.0 ** -RHO[t]
        assert np.array_equal(np.float16(f).astype(np.float64), f), t
    for same in ([(1, 2), (0, 3)], [(1, 3), (0, 4), (2, 2)]):  # one scale per shared accumulator
        assert len({RHO[a] + RHO[b] - int(E[a] + E[b]) for a, b in same}) == 1


def test_accumulators_of_dense_rows():
    n = 2048
    rng = np.random.default_rng(7)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    X = q[:, : n // 2] @ q[:, : n // 2].T
    rows = np.arange(0, n, 128)
    S = [s.astype(np.float64) for s in digits(X)]
    g = lambda a, b: S[a][rows] @ S[b].T  # noqa: E731
    exact = {"00": g(0, 0), "01": g(0, 1) + g(1, 0), "02": g(0, 2) + g(2, 0), "11": g(1, 1),
             "12+03": g(1, 2) + g(2, 1) + g(0, 3) + g(3, 0)}
    for k, v in exact.items():
        assert np.abs(v).max() < 2.0 ** 24, (k, np.log2(np.abs(v).max()))
    left = sum(g(a, b) * 2.0 ** -float(E[a] + E[b]) for a in range(5) for b in range(5) if a + b > 4)
    # seven 7-bit digits leave out (1, 6), (2, 5), (3, 4) and their mirrors: rms sqrt(6 K) 2^-52.6
    assert np.sqrt((left ** 2).mean()) < np.sqrt(6 * n) * 2.0 ** -52.6


@pytest.mark.gpu
@pytest.mark.parametrize("n", [17, 128, 129, 272, 1184, 2049, 2100])
def test_one_step_against_the_fp64_product(n):
    """One dense part: one tile, a full tile, one column more, a ragged split-K plan, and K beyond
    2048 (drained in two rounds).  The products left out have an rms of 0.8e-14 at K = 1,184
    and grow like sqrt(K); eight of them bound every element (less K than 1,184 is held to the same)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    H = (q * rng.uniform(-1.0, 1.0, n)) @ q.T
    H = 0.5 * (H + H.T)
    rowptr = np.arange(n + 1, dtype=np.int64) * n
    colind = np.tile(np.arange(n, dtype=np.int32), n)
    plan = gsp2.GSP2(n, rowptr, colind, n // 2, np.zeros(n, np.int32), 1, rowptr, colind, device="cuda:0",
                     precision="fp64e", ckpt_every=0, max_steps=1)
    got = plan.density(torch.from_numpy(H.ravel()).to("cuda:0"))
    alpha = plan.history()["alphas"][0]
    _, rep = plan.status()
    X = (rep["eps_max"] * np.eye(n) - H) / (rep["eps_max"] - rep["eps_min"])
    Y = X @ X
    want = 2.0 * X - Y if alpha > 0 else Y
    err = float(np.max(np.abs(plan.dense_p(got) - want)))
    print(f"n={n}: one step max|dX|={err:.2e}")
    assert err <= 8 * 0.8e-14 * max(1.0, np.sqrt(n / 1184))
