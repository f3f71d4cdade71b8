"""The work whose speed this repository looks after, as a list of cases.

A case is one call, or one training step, of a G-SP2 plan (paper_1801_10016_gb300.gsp2) on a
synthetic gapped tight-binding Hamiltonian: `sites` uniform in a cube at `density` sites per
cubic Angstrom, four orbitals per site (two near -8 eV, two near +2 eV), hopping
-exp(-r / 1.5) times a symmetric random 4 x 4 block between sites closer than 6 Angstrom,
`parts` parts by recursive coordinate bisection, and a dependency graph that joins orbitals
whose sites are closer than `radius`.  These are the sizes of the repository's workloads
(512 to 30,000 orbitals), and odd ones between them.  The geometry and with it the sparsity
pattern, the partition and the plan belong to the case, as in a molecular-dynamics or SCF run
that keeps its plan; the seed draws the values of H (and of the loss weights).

`op` is what the user does with the plan:
  density   P(H), the branch of every step chosen on the device;
  reuse     P of the next H of an SCF loop: the branches recorded for the previous H replayed,
            with the trace check and its host synchronisation;
  train     a training step: P through the autograd function, a loss linear in P, its gradient;
  refresh   the dependency graph of the next plan from the thresholded P.
"""

import functools
import math

import numpy as np
import torch

from paper_1801_10016_gb300 import gsp2

ORBS = 4
DENSE_PRECISIONS = ("fp64e", "fp16x3", "tf32x3", "bf16x3", "tf32", "bf16")


def listed():
    def c(name, op, precision, sites, parts, radius, density=0.1, uneven=False):
        return dict(name=name, op=op, precision=precision, sites=sites, parts=parts, radius=radius, density=density,
                    uneven=uneven)

    return [
        # the smallest problem with every option at its default (native FP64 steps): launches
        # and their latency
        c("tb512_fp64", "density", "fp64", 128, 8, 3.5),
        # one SCF iteration of a small molecule: replay, trace check, host synchronisation
        c("tb512_scf_fp64e", "reuse", "fp64e", 128, 8, 3.5),
        # odd counts of sites and parts, ragged tiles
        c("odd1044_fp64e", "density", "fp64e", 261, 7, 3.3),
        # training steps of the 4,096-orbital adjoint workload: FP64 results, and FP16-split
        # squarings with the FP32 adjoint
        c("tb4k_train_fp64e", "train", "fp64e", 1024, 32, 3.0),
        c("tb4k_train_fp16x3", "train", "fp16x3", 1024, 32, 3.0),
        # graph refresh between the plans of a long trajectory
        c("tb4k_refresh", "refresh", "fp64e", 1024, 32, 3.0),
        # plain BF16 squarings with FP64 refinement steps
        c("tb8k_bf16", "density", "bf16", 2000, 64, 5.0),
        # a training step whose parts fill the GPU, FP64 results
        c("tb8k_train_fp64e", "train", "fp64e", 2000, 64, 5.0),
        # dense molecular crystal: halos several times the core, the largest parts
        c("crystal8k_fp64e", "density", "fp64e", 2000, 64, 5.0, density=0.2),
        # very uneven parts (many small, a tail of large ones), TF32-split squarings, FP32 adjoint
        c("uneven12k_train_tf32x3", "train", "tf32x3", 3000, 102, 5.0, uneven=True),
        # the 30,000-orbital protein-sized workload: FP64 results, and the fastest precision
        # that passes the accuracy gates
        c("tb30k_fp64e", "density", "fp64e", 7500, 256, 5.0),
        c("tb30k_fp16x3", "density", "fp16x3", 7500, 256, 5.0),
    ]


def draw(rng):
    op = rng.choice(("density", "density", "reuse", "train", "train", "refresh"))
    top = {"density": 7000, "reuse": 5000, "train": 2400, "refresh": 1600}[op]
    sites = int(round(math.exp(rng.uniform(math.log(48), math.log(top)))))
    precision = "fp64e" if op in ("reuse", "refresh") else rng.choice(DENSE_PRECISIONS)
    if sites <= 700 and rng.random() < 0.2:
        precision = "fp64"  # native FP64 steps, as used on small problems
    parts = max(1, min(sites, int(round(sites / rng.uniform(14.0, 36.0)))))
    radius = round(rng.uniform(3.0, 5.0), 2)
    density = 0.1 if rng.random() < 0.8 or sites > 2000 else 0.2
    case = dict(op=op, precision=precision, sites=sites, parts=parts, radius=radius, density=density,
                uneven=rng.random() < 0.25)
    # no dearer than the largest listed case (the FP64 pipe is some 50 times slower)
    most = 4e10 if precision == "fp64" else 2.4e12
    while work(case)["flops"] > most:
        case["sites"] = case["sites"] * 4 // 5
        case["parts"] = max(1, case["parts"] * 4 // 5)
    return case


# ---------------------------------------------------------------- the problem behind a case


def _pairs(xyz, radius):
    """Site pairs a < b closer than `radius`, lexicographically, and their distances."""
    n = xyz.shape[0]
    out = []
    for a0 in range(0, n, 1024):
        d = ((xyz[a0:a0 + 1024, None, :] - xyz[None, :, :]) ** 2).sum(-1)
        a, b = torch.nonzero(d < radius * radius, as_tuple=True)
        keep = b > a + a0
        out.append((a[keep] + a0, b[keep], torch.sqrt(d[a[keep], b[keep]])))
    return tuple(torch.cat(q) for q in zip(*out))


def _csr(n, rows, cols):
    """CSR of the entries (rows, cols), and the place of each CSR entry in that list."""
    key, order = torch.sort(rows * n + cols)
    ptr = torch.searchsorted(key, n * torch.arange(n + 1, device=key.device))
    return ptr.cpu().numpy(), (key % n).to(torch.int32).cpu().numpy(), order


def _bisect(xyz, parts, weights):
    """Recursive coordinate bisection: sites split along the longest extent, each side in
    proportion to the weights of its parts."""
    part = np.empty(len(xyz), np.int32)
    cum = np.concatenate([[0.0], np.cumsum(weights)])
    todo = [(np.arange(len(xyz)), 0, parts)]
    while todo:
        idx, p0, m = todo.pop()
        if m == 1:
            part[idx] = p0
            continue
        ax = int(np.argmax(np.ptp(xyz[idx], axis=0)))
        idx = idx[np.lexsort((idx, xyz[idx, ax]))]
        left = m // 2
        cut = int(round(len(idx) * (cum[p0 + left] - cum[p0]) / (cum[p0 + m] - cum[p0])))
        cut = min(max(cut, left), len(idx) - (m - left))
        todo += [(idx[cut:], p0 + left, m - left), (idx[:cut], p0, left)]
    return part


@functools.lru_cache(maxsize=16)
def _geometry(sites, parts, radius, density, uneven):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rng = np.random.Generator(np.random.Philox(1234 + sites))
    xyz = rng.uniform(0.0, (sites / density) ** (1.0 / 3.0), size=(sites, 3))
    weights = 4.0 + 76.0 * rng.uniform(size=parts) ** 2 if uneven else np.ones(parts)
    part = np.repeat(_bisect(xyz, parts, weights), ORBS).astype(np.int32)
    t = torch.from_numpy(xyz).to(dev)
    n = ORBS * sites
    o = torch.arange(ORBS, device=dev)
    i, j = o[:, None].expand(ORBS, ORBS), o[None, :].expand(ORBS, ORBS)

    def block(a, b):  # orbital indices of the 4 x 4 blocks (a, b)
        return (ORBS * a[:, None, None] + i).reshape(-1), (ORBS * b[:, None, None] + j).reshape(-1)

    a, b, r = _pairs(t, 6.0)
    (ra, ca), (rb, cb) = block(a, b), block(b, a)
    diag = torch.arange(n, device=dev)
    rowptr, colind, order = _csr(n, torch.cat([ra, rb, diag]), torch.cat([ca, cb, diag]))
    ga, gb, _ = _pairs(t, radius)
    s = torch.arange(sites, device=dev)
    gr, gc = block(torch.cat([ga, gb, s]), torch.cat([gb, ga, s]))
    off = gr != gc
    g_rowptr, g_colind, _ = _csr(n, gr[off], gc[off])
    return dict(n=n, sites=sites, parts=parts, part=part, rowptr=rowptr, colind=colind, order=order, r=r, dev=dev,
                g_rowptr=g_rowptr, g_colind=g_colind)


def _geo(case):
    return _geometry(case["sites"], case["parts"], case["radius"], case["density"], case["uneven"])


def _h_values(geo, seed, shift=0.0):
    """Values of H on the pattern; `shift` > 0 mixes in that much of another draw (the H of a
    neighbouring SCF iteration)."""
    dev = geo["dev"]
    r = geo["r"]

    def one(s):
        g = torch.Generator(device=dev)
        g.manual_seed(s)
        on = torch.rand((geo["sites"], ORBS), dtype=torch.float64, device=dev, generator=g) - 0.5
        on[:, :2] -= 8.0
        on[:, 2:] += 2.0
        R = 2.0 * torch.rand((r.numel(), ORBS, ORBS), dtype=torch.float64, device=dev, generator=g) - 1.0
        blocks = (-torch.exp(-r / 1.5)[:, None, None] * 0.5 * (R + R.transpose(1, 2))).reshape(-1)
        return torch.cat([blocks, blocks, on.reshape(-1)])[geo["order"]]

    v = one(seed)
    return v if shift == 0.0 else (1.0 - shift) * v + shift * one(seed + 7919)


def _weights(geo, seed, count):
    """Loss weights of a training step, one per stored value of P."""
    g = torch.Generator(device=geo["dev"])
    g.manual_seed(seed + 104729)
    return torch.randn(count, dtype=torch.float64, device=geo["dev"], generator=g)


# ---------------------------------------------------------------- what is measured


def prepare(case, seed):
    geo = _geo(case)
    adjoint = 8 if case["op"] == "train" else 0
    plan = gsp2.GSP2(geo["n"], geo["rowptr"], geo["colind"], 2 * geo["sites"], geo["part"], geo["parts"],
                     geo["g_rowptr"], geo["g_colind"], precision=case["precision"], ckpt_every=adjoint)
    h = _h_values(geo, seed)
    state = dict(op=case["op"], plan=plan, h=h)
    if case["op"] == "reuse":
        # the SCF loop's previous iteration recorded the branches
        alpha = torch.zeros(plan.alpha_len, dtype=torch.int8, device=h.device)
        state["nsteps"] = plan.density_reuse(_h_values(geo, seed, shift=1e-3), alpha, 0)[1]
        state["alpha"] = alpha
    elif case["op"] == "train":
        state["weights"] = _weights(geo, seed, plan.nnz_p)
        h.requires_grad_(True)
    elif case["op"] == "refresh":
        state["p"] = plan.density(h)
        # room for the graph at any threshold: its columns come back in an array of one size
        state["columns"] = np.empty(len(plan.threshold_graph(state["p"], 0.0)[1]), np.int32)
    return state


def run(state):
    plan, h = state["plan"], state["h"]
    if state["op"] == "density":
        return plan.density(h)
    if state["op"] == "reuse":
        p, state["nsteps"], _, status = plan.density_reuse(h, state["alpha"], state["nsteps"])
        return {"p": p, "nsteps": state["nsteps"], "status": status}
    if state["op"] == "train":
        h.grad = None
        p = gsp2.gsp2_density(h, plan)
        (state["weights"] * p).sum().backward()
        return {"p": p.detach(), "grad": h.grad}
    rowptr, colind = plan.threshold_graph(state["p"], 1e-5)
    state["columns"][:len(colind)] = colind
    state["columns"][len(colind):] = -1
    return {"rowptr": rowptr, "columns": state["columns"]}


# ---------------------------------------------------------------- what it cannot do without


def _members(geo):
    """Per part its vertices (cores ascending, then the halo ascending) and its core count."""
    part, ptr, col = geo["part"], geo["g_rowptr"], geo["g_colind"]
    out = []
    by_part = np.argsort(part, kind="stable")
    ends = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=geo["parts"]))])
    rows = np.repeat(np.arange(geo["n"]), np.diff(ptr))
    cross = part[rows] != part[col]
    kp, kv = part[rows[cross]].astype(np.int64), col[cross].astype(np.int64)
    halo = np.unique(kp * geo["n"] + kv)
    hend = np.searchsorted(halo, np.arange(geo["parts"] + 1) * geo["n"])
    for k in range(geo["parts"]):
        core = by_part[ends[k]:ends[k + 1]]
        out.append((np.concatenate([core, halo[hend[k]:hend[k + 1]] % geo["n"]]), len(core)))
    return out


STEPS = 18  # purification steps of a gapped system of this kind (17 to 23)


def work(case):
    geo = _geo(case)
    s = np.array([len(v) for v, _ in _members(geo)], np.float64)
    c = np.array([m for _, m in _members(geo)], np.float64)
    nnz_h, nnz_p = float(geo["rowptr"][-1]), float((c * s).sum())
    square = float((s * s * (s + 1.0)).sum())  # one symmetric square of every part
    if case["op"] == "refresh":
        # every stored value of P read once; the graph (at most its pattern) written once
        return {"bytes": 8.0 * nnz_p + 4.0 * nnz_p + 8.0 * geo["n"], "flops": nnz_p}
    if case["op"] == "train":
        # P and the gradient: the squares, then two symmetric products per reverse step
        return {"bytes": 16.0 * nnz_h + 16.0 * nnz_p, "flops": 3.0 * STEPS * square}
    return {"bytes": 8.0 * nnz_h + 8.0 * nnz_p, "flops": STEPS * square}


# ---------------------------------------------------------------- the same in 64 bits


def exact(case, seed):
    """G-SP2 in plain 64-bit torch: global Gershgorin bounds, one branch for all parts per step
    from the summed core traces, the idempotency stopping test, two alternating steps after it
    for the low-precision plans, core columns into P; for a training step the reverse sweep
    through the same branches."""
    if case["op"] == "refresh":
        return None
    geo = _geo(case)
    dev, n = geo["dev"], geo["n"]
    v = _h_values(geo, seed)
    rows = torch.from_numpy(np.repeat(np.arange(n), np.diff(geo["rowptr"]))).to(dev)
    cols = torch.from_numpy(geo["colind"].astype(np.int64)).to(dev)
    on = rows == cols
    centre = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, rows[on], v[on])
    radius = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, rows[~on], v[~on].abs())
    lo, hi = float((centre - radius).min()), float((centre + radius).max())
    members = _members(geo)
    train = case["op"] == "train"
    loc = torch.full((n,), -1, dtype=torch.int64, device=dev)
    X, S = [], []
    for verts, _ in members:
        idx = torch.from_numpy(verts).to(dev)
        S.append(idx)
        loc[idx] = torch.arange(len(verts), device=dev)
        ptr = torch.from_numpy(geo["rowptr"]).to(dev)
        cnt = ptr[idx + 1] - ptr[idx]
        at = torch.arange(int(cnt.sum()), device=dev) + torch.repeat_interleave(
            ptr[idx] - torch.cumsum(cnt, 0) + cnt, cnt)
        li = torch.repeat_interleave(torch.arange(len(verts), device=dev), cnt)
        lj = loc[cols[at]]
        keep = lj >= 0
        x = torch.zeros((len(verts), len(verts)), dtype=torch.float64, device=dev)
        x[li[keep], lj[keep]] = -v[at][keep]
        x.diagonal().add_(hi)
        X.append(x / (hi - lo))
        loc[idx] = -1
    nocc = 2 * geo["sites"]
    core = [c for _, c in members]
    its, alphas, idem = [X], [], []
    trace = sum(float(x.diagonal()[:c].sum()) for x, c in zip(X, core))
    tail = 0 if case["precision"] in ("fp64", "fp64e") else 2
    left = -1
    while True:
        if left >= 0:
            a = -alphas[-1] if left < tail else (1 if trace <= nocc else -1)
        else:
            a = 1 if trace <= nocc else -1
        new, sq, tn = [], 0.0, 0.0
        for x, c in zip(X, core):
            y = x @ x
            sq += float(y.diagonal()[:c].sum())
            y = 2.0 * x - y if a > 0 else y
            tn += float(y.diagonal()[:c].sum())
            new.append(y)
        idem.append(trace - sq)
        alphas.append(a)
        X, trace = new, tn
        if train:
            its.append(X)
        if left >= 0:
            left -= 1
            if left == 0:
                break
            continue
        i = len(alphas)
        e = idem[-1]
        if (i >= 2 and abs(e) <= 1e-3 and (e < 0 or e >= idem[-2])) or i == 45:
            if tail == 0:
                break
            left = tail
    p, _ = _p_vector(geo, members, X)
    if case["op"] == "reuse":
        return {"p": p, "nsteps": None, "status": None}
    if not train:
        return p
    w = _weights(geo, seed, p.numel())
    grad = torch.zeros((n, n), dtype=torch.float64, device=dev)
    seeds = _p_matrices(geo, members, w)
    for k, (idx, c) in enumerate(zip(S, core)):
        g = torch.zeros((len(idx), len(idx)), dtype=torch.float64, device=dev)
        g[:, :c] = seeds[k]
        g = 0.5 * (g + g.T)
        for i in range(len(alphas), 0, -1):
            x = its[i - 1][k]
            z = g @ x
            z = z + z.T
            g = 2.0 * g - z if alphas[i - 1] > 0 else z
        grad[idx[:, None], idx[None, :]] -= g / (hi - lo)
    return {"p": p, "grad": grad[rows, cols]}


def _columns(geo, members):
    """For each part: the start in P's value array of each of its core columns, and the order
    that sorts its vertices (the rows of each column ascend)."""
    size = np.empty(geo["n"], np.int64)
    for verts, c in members:
        size[verts[:c]] = len(verts)
    ptr = np.concatenate([[0], np.cumsum(size)])
    return ptr, [(ptr[verts[:c]], np.argsort(verts, kind="stable")) for verts, c in members]


def _p_vector(geo, members, X):
    ptr, where = _columns(geo, members)
    p = torch.empty(int(ptr[-1]), dtype=torch.float64, device=geo["dev"])
    for (start, order), x, (verts, c) in zip(where, X, members):
        at = torch.from_numpy(start[:, None] + np.arange(len(verts))[None, :]).to(geo["dev"])
        p[at] = x[:, :c].T[:, torch.from_numpy(order).to(geo["dev"])]
    return p, ptr


def _p_matrices(geo, members, p):
    """The inverse of _p_vector: per part the s x c matrix of its core columns."""
    _, where = _columns(geo, members)
    out = []
    for (start, order), (verts, c) in zip(where, members):
        at = torch.from_numpy(start[:, None] + np.arange(len(verts))[None, :]).to(geo["dev"])
        m = torch.empty((len(verts), c), dtype=torch.float64, device=geo["dev"])
        m[torch.from_numpy(order).to(geo["dev"])] = p[at].T
        out.append(m)
    return out
