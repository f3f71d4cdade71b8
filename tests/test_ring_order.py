"""The rings of operand tiles of the emulated step, as a model on the CPU: two producers (rows I, rows J)
fill the places in turn, the issuing warp releases them step by step as oz_step_kernel does, and the barriers show a
phase by its parity only.  No place may be filled while its tile is still needed, and the walk must end, whatever
the speed of the warps and in whatever order the releases of one step become visible (those of a later
step follow: its MMAs end later).

The rings have an odd number of places, so that a place changes its owner every lap and a producer sees every second
phase of it: it may wait for a place when its turn comes, but not look at places further on, where
the phase before the one it waits for, of the same parity as the one before that, can still be open."""

import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_10016_gb300", "csrc")


def wide_slice(T, dg):
    """Places of a wide slice of T digits: [(operand, tile)], the places each step releases, and the waits of the MMA
    warp: its first group of places, and the group to wait for before a step's last MMAs."""
    order = [(0, T - 1 - i) for i in range(T)] if dg else [(op, (T - 1 - i) if op == 0 else i)
                                                             for i in range(T) for op in (0, 1)]
    at = {v: k for k, v in enumerate(order)}
    rel = {i: [] for i in range(T)}
    if dg:
        rel[T - 1] = list(range(T))
        return order, rel, list(range(T)), {}
    for i in range(T):
        q = T - 1 - i
        lo = 2 - q if T == 5 and q < 2 else 0
        rel[i].append(at[(0, q)])
        for b in range(lo, i + 1):
            later = any((2 - (T - 1 - m) if T == 5 and T - 1 - m < 2 else 0) <= b <= m for m in range(i + 1, T))
            if not later:
                rel[i].append(at[(1, b)])
    return order, rel, list(range(6 if T == 5 else 4)), ({2: list(range(6, 10))} if T == 5 else {})


def narrow_slice(dg):
    return [(0, 0)] if dg else [(0, 0), (1, 0)], {0: [0] if dg else [0, 1]}, list(range(1 if dg else 2)), {}


def items(rng, wide):
    out = []
    for _ in range(rng.randint(2, 5)):
        dg, n = rng.random() < 0.4, rng.randint(1, 6)
        if wide:
            out.append((dg, [wide_slice(5, dg)] * n + [wide_slice(2, dg)] * n))
        else:
            out.append((dg, [narrow_slice(dg)] * (n + (n + 1) // 2)))
    return out


def run(rng, places, work, ahead):
    phase, live, loaded, pending, bad = [0] * places, [None] * places, set(), [], []
    published = [0]  # items that warp 0 (rows I) has passed on: after all its loads of the one before
    starts, flat, pos = [], [], 0
    for dg, sl in work:
        starts.append(len(flat))
        for s in sl:
            flat.append((dg, pos, *s))
            pos += len(s[0])

    def done(x):
        return phase[x % places] % 2 == (x // places) % 2

    def producer(op):
        for v, (dg, sl) in enumerate(work):
            if op == 0:
                published[0] = v + 1
            while published[0] <= v:
                yield False
            if dg and op == 1:
                continue
            for n in range(starts[v], starts[v] + len(sl)):
                _, base, order, *_ = flat[n]
                mine = [base + k for k, (o, _) in enumerate(order) if o == op]
                ready = {x for x in mine[:ahead] if done(x)}
                yield True
                for x in mine:
                    while x not in ready and not done(x):
                        yield False
                    if live[x % places] is not None:
                        bad.append(x)
                    live[x % places] = x
                    loaded.add(x)
                    yield True

    def mma():
        def has(n, group):
            return all(flat[n][1] + k in loaded for k in group)
        while not has(0, flat[0][4]):
            yield False
        for n, (dg, base, order, rel, first, groups) in enumerate(flat):
            for i in sorted(rel):
                while i in groups and not has(n, groups[i]):
                    yield False
                last_of_item = n + 1 == len(flat) or n + 1 in starts
                if i == max(rel) and not last_of_item:
                    while not has(n + 1, flat[n + 1][4]):
                        yield False
                if rel[i]:
                    pending.append([base + k for k in rel[i]])
                yield True
            if n + 1 < len(flat):
                while not has(n + 1, flat[n + 1][4]):
                    yield False

    def releases():
        while True:
            if not pending:
                yield False
                continue
            x = pending[0].pop(rng.randrange(len(pending[0])))
            if not pending[0]:
                pending.pop(0)
            live[x % places] = None
            phase[x % places] += 1
            yield True

    tasks, left, idle = [producer(0), producer(1), mma(), releases()], {0, 1, 2}, 0
    weight = [rng.random() ** 2 + 0.02 for _ in tasks]
    while left:
        t = rng.choices(range(4), weight)[0]
        if t < 3 and t not in left:
            continue
        try:
            moved = next(tasks[t])
        except StopIteration:
            left.discard(t)
            moved = True
        if bad:
            return "overwritten"
        idle = 0 if moved else idle + 1
        if idle > 20000:
            return "stuck"
    return "ok"


@pytest.mark.parametrize("wide,places", [(True, 13), (False, 5)])
def test_waiting_in_turn_never_overwrites(wide, places):
    for seed in range(400):
        rng = random.Random(seed)
        assert run(rng, places, items(rng, wide), ahead=0) == "ok", seed


def test_looking_ahead_would():
    assert any(run(rng, 13, items(rng, True), ahead=5) == "overwritten" for rng in map(random.Random, range(400)))


def test_the_kernel_has_these_rings_and_waits_in_turn():
    src = open(os.path.join(CSRC, "k_oz.cu")).read()
    assert "constexpr int OZ_TILES = 13;" in src and "constexpr int OZ_UNITS = 5;" in src
    kernel = src[src.index("oz_step_kernel(const"):src.index("cudaError_t launch_oz_convert")]
    assert len(re.findall(r"mbar_test\(", kernel)) == 0


@pytest.mark.gpu
def test_wide_plan_repeats():
    """The adjoint of one part of 3,900 orbitals (496 tiles in wide slices), over and over: an overwritten digit tile
    shows as a 128 x 128 block of Xbar off by 1e-6.  The runs differ by no more than rounding (the scales come from
    sums in FP32 by atomics)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1801_10016_gb300 import gsp2
    from synth import make_tb_system
    s = make_tb_system(975, 1, 3.0, seed=71)
    plan = gsp2.GSP2(s.n, s.rowptr, s.colind, s.nocc, s.part, s.nparts, s.g_rowptr, s.g_colind, device="cuda:0",
                     ckpt_every=4, precision="fp64e")
    h = torch.from_numpy(s.vals).to("cuda:0")
    torch.manual_seed(3)
    pb = torch.randn(plan.nnz_p, dtype=torch.float64, device="cuda:0")
    p0 = h0 = None
    worst = 0.0
    for _ in range(100):
        p = plan.density(h)
        hb = plan.backward(pb)
        if p0 is None:
            p0, h0 = p.clone(), hb.clone()
        assert torch.equal(p, p0)
        worst = max(worst, float((hb - h0).abs().max()))
    print(f"largest difference between runs {worst:.1e}")
    assert worst <= 1e-10
