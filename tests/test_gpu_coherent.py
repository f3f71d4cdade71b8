"""Emulated FP64 steps on rows whose digits are coherent (entries of one magnitude, or slowly
varying), where the sums of digit products pass 2^24 in FP32: the purification of a Hadamard matrix and
of a half-filled ring, and an adjoint seed of one value, each step against the FP64 product.

Tolerance of one step, from its definition alone (nothing is allowed for the accumulation of the products
that are to be exact): the products left out, from the digits themselves; the digits' remainder, at most
2^-50 + 2^-57 an entry on either factor; and for every 32 columns 2^-57 of each of two roundings to the fixed
point, and as much again for the sixth accumulator, whose sums over 16 columns have an ulp below 2^-56.  The
rounding of the FP64 product, of the order of sqrt(n) 2^-53, is allowed for as well; the forward steps are held
against an exact one, since the sums of equal terms round all in one direction."""

import numpy as np
import pytest

WIDTHS = (11, 8, 11, 8, 11)
E = [int(e) for e in np.cumsum(WIDTHS)]


def hadamard(n):
    H = np.ones((1, 1))
    while H.shape[0] < n:
        H = np.block([[H, H], [H, -H]])
    return H / np.sqrt(n)


def ring(n):
    H = np.zeros((n, n))
    k = np.arange(n)
    H[k, (k + 1) % n] = H[(k + 1) % n, k] = -1.0
    return H


def digits(x):
    """S_0 .. S_4 of a float64 tensor (x 2^49 is exact), as in test_digit_products."""
    import torch
    r = torch.round(x * 2.0 ** E[-1]).to(torch.int64)
    S = [None] * 5
    for t in range(4, 0, -1):
        b = 1 << WIDTHS[t]
        S[t] = torch.remainder(r + b // 2, b) - b // 2
        r = torch.div(r - S[t], b, rounding_mode="floor")
    S[0] = r
    return [s.to(torch.float64) for s in S]


EXACT = [((0, 0),), ((0, 1), (1, 0)), ((0, 2), (2, 0)), ((1, 1),), ((1, 2), (2, 1), (0, 3), (3, 0))]


def sums(A, B, rows):
    """Largest sum of the exact accumulators for A B^T on the sampled rows, and the products left out."""
    top = max(float(sum(A[a][rows] @ B[b].T for a, b in g).abs().max()) for g in EXACT)
    left = sum(A[a][rows] @ B[b].T * 2.0 ** -float(E[a] + E[b]) for a in range(5) for b in range(5) if a + b > 4)
    return top, float(left.abs().max())


def exact_square(x):
    """x x for a symmetric x on the grid 2^-56, |x| <= 1: three digits of 19 bits, whose products add up
    exactly in FP64 (n 2^36 < 2^53), then rounded once per digit pair from the smallest up."""
    import torch
    d0 = torch.round(x * 2.0 ** 18)
    r = x * 2.0 ** 18 - d0
    d1 = torch.round(r * 2.0 ** 19)
    d2 = (r * 2.0 ** 19 - d1) * 2.0 ** 19
    assert bool((d2 == torch.round(d2)).all())
    y = (d2 @ d2) * 2.0 ** -112
    m = d1 @ d2
    y += (m + m.T) * 2.0 ** -93
    m = d0 @ d2
    y += (m + m.T + d1 @ d1) * 2.0 ** -74
    m = d0 @ d1
    y += (m + m.T) * 2.0 ** -55
    return y + (d0 @ d0) * 2.0 ** -36


def step_bound(X, left):
    n = X.shape[0]
    one = float(X.abs().sum(1).max())
    return left + 2 * one * (2.0 ** -50 + 2.0 ** -57) + (n / 32 + 1) * 4 * 2.0 ** -57 + np.sqrt(n) * 2.0 ** -53


def test_rounds_of_32_are_exact():
    """Sums over 32 columns stay below 2^24 for any X with 0 <= X <= 1, from the digits' ranges: a row's
    off-diagonal 2-norm is at most (x_ii - x_ii^2)^(1/2), so 32 of its entries sum to at most (1 + sqrt(33)) / 2."""
    s0 = 2.0 ** 11 * (1 + np.sqrt(33.0)) / 2 + 32 / 2.0  # sum of |S_0|, each within 1/2 of 2^11 |x|
    h = {1: 2.0 ** 7, 2: 2.0 ** 10, 3: 2.0 ** 7}  # |S_t|
    assert 2 * s0 * h[1] < 2.0 ** 24 and 2 * s0 * h[2] < 2.0 ** 24 and 32 * h[1] ** 2 < 2.0 ** 24
    assert 2 * s0 * h[3] + 2 * 32 * h[1] * h[2] < 2.0 ** 24
    # the adjoint: rows of Xbar / 2^sig have 2-norm <= 1/2
    sb = 2.0 ** 11 * np.sqrt(32.0) / 2 + 32 / 2.0
    assert (s0 + sb) * h[2] < 2.0 ** 24 and (s0 + sb) * h[3] + 2 * 32 * h[1] * h[2] < 2.0 ** 24


def dense_plan(n, steps, **kw):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    rowptr = np.arange(n + 1, dtype=np.int64) * n
    colind = np.tile(np.arange(n, dtype=np.int32), n)
    return gsp2.GSP2(n, rowptr, colind, n // 2, np.zeros(n, np.int32), 1, np.zeros(n + 1, np.int64),
                     np.zeros(0, np.int32), device="cuda:0", precision="fp64e", max_steps=steps, fp64_tail_steps=0, **kw)


# one K half an item and 64-column pieces; the same unsplit; whole tiles; rounds of 2,048 in wide slices; ragged
@pytest.mark.parametrize("matrix,n,split,steps", [("hadamard", 512, -1, (3, 9)), ("hadamard", 512, 0, (3, 9)),
                                                  ("hadamard", 2048, -1, (3, 9)), ("hadamard", 4096, -1, (3, 6)),
                                                  ("ring", 1500, -1, (29, 34))])
@pytest.mark.gpu
def test_steps_whose_sums_pass_2_24(matrix, n, split, steps):
    import torch
    H = -hadamard(n) if matrix == "hadamard" else ring(n)
    plan = dense_plan(n, 40, split_k=split, ckpt_every=0)
    h = torch.from_numpy(H.ravel()).to("cuda:0")
    plan.density(h)
    alphas = plan.history()["alphas"][:steps[1] + 1]
    alpha = torch.zeros(plan.alpha_len, dtype=torch.int8, device="cuda:0")
    alpha[:len(alphas)] = torch.tensor(alphas, dtype=torch.int8)
    x0, worst, most = None, 0.0, 0.0
    for m in range(steps[0], len(alphas) + 1):  # X_m by a replay of m steps
        p = plan.density(h, alpha=alpha, mode="replay", nsteps=m)
        x1 = torch.from_numpy(plan.dense_p(p)).to("cuda:0")
        if x0 is not None:
            y = exact_square(x0)
            want = 2 * x0 - y if alphas[m - 1] > 0 else y
            S = digits(x0)
            top, left = sums(S, S, slice(None))
            err, tol = float((x1 - want).abs().max()), step_bound(x0, left)
            print(f"{matrix} n={n} step {m}: largest sum 2^{np.log2(top):.1f}, left out {left:.1e}, max|dX| {err:.2e} of {tol:.2e}")
            worst, most = max(worst, err / tol), max(most, top)
        x0 = x1
    p2 = plan.density(h, alpha=alpha, mode="replay", nsteps=len(alphas))
    assert torch.equal(p, p2)  # whichever blocks formed the part again
    assert most >= 2.0 ** 24
    assert worst <= 1.0


@pytest.mark.gpu
@pytest.mark.parametrize("n", [600, 1500, 4000])
def test_reverse_step_on_a_seed_of_one_value(n):
    """Hbar of one step with H and Pbar of one magnitude and the same signs: -(Xbar X + X Xbar) (or 2 Xbar
    less that) over the width of the bounds."""
    import torch
    sign = np.where((np.arange(n)[:, None] // 7 + np.arange(n)[None, :] // 7) % 2, 1.0, -1.0)
    H = 0.31 * sign
    plan = dense_plan(n, 1, ckpt_every=1)
    h = torch.from_numpy(H.ravel()).to("cuda:0")
    plan.density(h)
    alpha = plan.history()["alphas"][0]
    _, rep = plan.status()
    pb = torch.from_numpy(0.7313 * sign).to("cuda:0")
    got = plan.backward(pb.reshape(-1).contiguous()).reshape(n, n)
    width = rep["eps_max"] - rep["eps_min"]
    X = (rep["eps_max"] * torch.eye(n, dtype=torch.float64, device="cuda:0") - h.reshape(n, n)) / width
    Z = pb @ X + X @ pb
    want = -(2 * pb - Z if alpha > 0 else Z) / width
    sig = int(np.ceil(np.log2(2 * float(pb.norm(dim=1).max()) * (1 + 2.0 ** -20))))
    rows = torch.arange(0, n, n // 16 + 1, device="cuda:0")
    sx, sb = digits(X), digits(pb * 2.0 ** -sig)
    t0, l0 = sums(sb, sx, rows)
    t1, l1 = sums(sx, sb, rows)
    one = float(X.abs().sum(1).max() + (pb * 2.0 ** -sig).abs().sum(1).max())
    tol = (l0 + l1 + 2 * one * (2.0 ** -50 + 2.0 ** -57) + (2 * n / 32 + 2) * 4 * 2.0 ** -57
           + np.sqrt(2 * n) * 2.0 ** -53) * 2.0 ** sig / width
    err = float((got - want).abs().max())
    print(f"n={n}: sums 2^{np.log2(t0 + t1):.1f}, left out {(l0 + l1):.1e}, max|dHbar| {err:.2e} of {tol:.2e}")
    assert t0 + t1 >= 2.0 ** 24
    assert err <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("split", [-1, 1])
def test_one_coherent_part_among_others(split):
    """A ring of 1,500 in one part beside six gapped blocks of 160 in parts of their own: P and Hbar against the
    native FP64 path on the same branches (the parts formed again and rebuilt among the others), and the same bits
    for claimed and dealt items, either order, and launches without a graph."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    rng = np.random.default_rng(12)
    sizes = [160, 160, 160, 1500, 160, 160, 160]
    blocks = []
    for m in sizes:
        if m == 1500:
            blocks.append(ring(m))
        else:
            b = rng.standard_normal((m, m)) * 0.02
            blocks.append(np.diag(np.where(np.arange(m) % 2, 1.2, -1.2)) + 0.5 * (b + b.T))
    n = sum(sizes)
    starts = np.concatenate([[0], np.cumsum(sizes)])
    part = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    rowptr = np.concatenate([[0], np.cumsum(np.repeat(sizes, sizes))]).astype(np.int64)
    colind = np.concatenate([np.arange(starts[k], starts[k + 1]) for k, m in enumerate(sizes) for _ in range(m)]).astype(np.int32)
    h = torch.from_numpy(np.concatenate([b.ravel() for b in blocks])).to("cuda:0")

    def make(precision, **kw):
        return gsp2.GSP2(n, rowptr, colind, n // 2, part, len(sizes), np.zeros(n + 1, np.int64), np.zeros(0, np.int32),
                         device="cuda:0", precision=precision, max_steps=36, fp64_tail_steps=0, ckpt_every=5, **kw)

    plan = make("fp64e", split_k=split)
    p = plan.density(h)
    alphas = plan.history()["alphas"]
    torch.manual_seed(5)
    pb = torch.randn(plan.nnz_p, dtype=torch.float64, device="cuda:0")
    hb = plan.backward(pb)
    alpha = torch.zeros(plan.alpha_len, dtype=torch.int8, device="cuda:0")
    alpha[:len(alphas)] = torch.tensor(alphas, dtype=torch.int8)
    ref = make("fp64")
    want = ref.density(h, alpha=alpha, mode="replay", nsteps=len(alphas))
    want_h = ref.backward(pb)
    err, err_h = float((p - want).abs().max()), float((hb - want_h).abs().max())
    scale = max(1.0, float(want_h.abs().max()))
    print(f"split {split}: {len(alphas)} steps, max|dP| {err:.1e}, max|dHbar| {err_h:.1e} of {scale:.1e}")
    assert err <= 1e-10 and err_h <= 1e-9 * scale
    for kw in (dict(tile_claim=0), dict(tile_order=0), dict(use_graph=0)):
        other = make("fp64e", split_k=split, **kw)
        assert torch.equal(other.density(h), p), kw
        assert torch.equal(other.backward(pb), hb), kw
