"""What a user of this framework has it do, as cases that can be timed and compared.

A case names an operation, the size of the particle set, the octree depth, the
refinement constant and the options of the call:

  field      the whole path on device-resident particles: tree, operators,
             deposit, Poisson solve, gather
  tree       node selection for a new particle set (every time step builds one)
  operators  neighbour search, WLS operators and matrices on a node set, then
             both assembled matrices applied once
  solve      the Poisson solve on an assembled system
  batch      the same for a batch of independent beams
  gather     derivatives at the nodes and potential and field at the particles
  vp         one leapfrog step with its new field solve
  train      one training step of the learned preconditioner on a new system

Particles follow the beam-with-halo law in random order (drawn again inside their
deepest cells for every seed).  Sizes: the benchmark
workloads (1e5 particles at depth 6, 1e7 at depth 10, 64 beams at depth 9), the
profiled ones (2e6 and 2e7 particles at depth 9), the training systems (1e5
particles at depth 8) and the tests' beams.
"""
import math

import numpy as np
import torch

from paper_1603_04039_gb300 import APCloud, MPNN, VlasovPoisson, inputs

DEV = "cuda:0"
# FP64 solves run to the tolerance of the parity tests, the benchmark workloads
# to the benchmark's, the other mixed-form solves to that of the mixed tests
RTOL = {"fp64": 1e-12, "mixed": 1e-11, "bench": 1e-10}
MAX_ITER = 20000


def listed():
    return [
        # a small beam solved from particles to field with the default options:
        # launches and host waits are most of it
        dict(name="field_1e5_fp64", op="field", n=100_000, depth=6, c=1.0, precision="fp64", degree=1, tol="fp64"),
        # the benchmark's own workload: mixed form, degree-16 polynomial, tuned launch shape
        dict(name="field_1e7_mixed", op="field", n=10_000_000, depth=10, c=0.043, precision="mixed", degree=16,
             tol="bench"),
        # node selection of a training-size beam and of the largest particle set
        dict(name="tree_1e5", op="tree", n=100_000, depth=8, c=0.15),
        dict(name="tree_2e7", op="tree", n=20_000_000, depth=9, c=0.15),
        # operators in the default FP64 form (a test-size system) and in the
        # mixed form (an adaptive beam of a few 1e5 nodes)
        dict(name="operators_2e5_fp64", op="operators", n=200_000, depth=8, c=0.1, precision="fp64"),
        dict(name="operators_2e6_mixed", op="operators", n=2_000_000, depth=9, c=0.043, precision="mixed"),
        # Poisson solves: plain FP64 GMRES(30) with Jacobi, and the mixed form
        # on a system that fits in L2
        dict(name="solve_1e5_fp64", op="solve", n=100_000, depth=8, c=0.15, precision="fp64", degree=1, tol="fp64"),
        dict(name="solve_1e6_mixed", op="solve", n=1_000_000, depth=8, c=0.08, precision="mixed", degree=16,
             tol="mixed"),
        # 64 beams of 1e4 to 1e6 particles solved together (4.8e6 nodes)
        dict(name="batch_64_mixed", op="batch", beams=64, n_lo=10_000, n_hi=1_000_000, depth=9, c=0.05,
             precision="mixed", degree=16, tol="bench"),
        # field of the most particles on few nodes
        dict(name="gather_2e7_mixed", op="gather", n=20_000_000, depth=9, c=0.15, precision="mixed"),
        # a time step of a million-particle beam, warm-started
        dict(name="vp_1e6_mixed", op="vp", n=1_000_000, depth=8, c=0.08, precision="mixed", degree=16, tol="bench"),
        # a training step: system, loss, gradients, Adam
        dict(name="train_1e5", op="train", n=100_000, depth=8, c=0.15),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _beam(rng, n_lo, n_hi, nodes_lo, nodes_hi):
    """Particle count, depth and refinement constant for a node count in the range.
    The criterion gives about 1.35 (N / c^2)^0.6 nodes; the depth lets the core refine fully."""
    n = int(_log(rng, n_lo, n_hi))
    nodes = _log(rng, nodes_lo, min(nodes_hi, 0.5 * n))
    c = round(math.sqrt(n / (nodes / 1.35) ** (1 / 0.6)), 4)
    core = 0.9 / (0.05 * math.sqrt(2 * math.pi)) ** 3
    depth = math.ceil(math.log2(2.0 / (c * c / (core * n)) ** 0.2))
    return n, max(4, min(10, depth)), c


def draw(rng):
    op = rng.choice(["field", "tree", "operators", "solve", "solve", "batch", "gather", "vp", "train"])
    prec = rng.choice(["fp64", "mixed"])
    case = dict(op=op)
    if op == "tree":
        case["n"], case["depth"], case["c"] = _beam(rng, 1e4, 2e7, 600, 1e6)
    elif op == "operators":
        case["n"], case["depth"], case["c"] = _beam(rng, 1e4, 1e7, 600, 5e4 if prec == "fp64" else 1e6)
        case["precision"] = prec
    elif op == "gather":
        case["n"], case["depth"], case["c"] = _beam(rng, 1e4, 2e7, 600, 5e5)
        case["precision"] = prec
    elif op == "batch":
        lo = int(_log(rng, 1e4, 1e5))
        case.update(beams=rng.randint(2, 64), n_lo=lo, n_hi=lo * rng.randint(2, 10), depth=rng.randint(6, 9),
                    c=round(_log(rng, 0.06, 0.5), 4), precision="mixed", degree=16, tol="mixed")
    elif op == "train":
        case["n"], case["depth"], case["c"] = _beam(rng, 2e4, 2e5, 2e3, 3e4)
    else:
        poly = prec == "mixed" or rng.random() < 0.4
        most = {"vp": 2e5, "field": 1e6, "solve": 1e6}[op] if prec == "mixed" else (1e5 if poly else 2e4)
        if op == "vp":
            prec, poly, most = "mixed", True, 2e5
        case["n"], case["depth"], case["c"] = _beam(rng, 1e4, 1e7 if op != "vp" else 2e6, 600, most)
        case.update(precision=prec, degree=16 if poly else 1, tol=prec)
    return case


# ---------------------------------------------------------------- inputs
def _particles(n, depth, seed, law_seed=1, **law):
    """A beam whose deepest cells hold the same numbers of particles for every seed, so that
    node counts (and the shapes of the outputs) do not change with it; the seed draws the
    places inside the cells, one of the cube's 48 symmetries and the order."""
    x, y, z, q = inputs.beam_with_halo_device(n, law_seed, DEV, **law)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    half = 2.0 ** (depth - 1)
    cell = torch.clamp(torch.floor((torch.stack([x, y, z]) + 1.0) * half), max=2 * half - 1)
    pos = (cell + 0.0005 + 0.999 * torch.rand(3, n, generator=g, device=DEV, dtype=torch.float64)) / half - 1.0
    order = torch.randperm(n, generator=g, device=DEV)
    kind = int(torch.randint(48, (1,), generator=g, device=DEV))
    axes = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)][kind >> 3]
    return tuple((pos[a] if kind >> d & 1 else -pos[a])[order] for d, a in enumerate(axes)) + (q,)


def _context(case):
    ap = APCloud(max_depth=case["depth"], c_refine=case["c"], precision=case.get("precision", "fp64"),
                 poly_degree=case.get("degree", 1), poly_omega=1.0 if case.get("degree", 1) > 1 else 0.7, device=DEV)
    if case.get("degree", 1) > 1:
        ap.set_launch_shape(256, 4, 4, 1)   # what the autotuner picks on the benchmark workloads
    return ap


def prepare(case, seed):
    op = case["op"]
    st = dict(case=case, rtol=RTOL[case.get("tol", "fp64")])
    if op == "batch":
        laws = inputs.beam_batch_params(case["beams"], 1, case["n_lo"], case["n_hi"])
        parts = [_particles(p["n"], case["depth"], 1000 * seed + p["seed"], p["seed"], sigma=p["sigma"],
                            halo_frac=p["halo_frac"], r0=p["r0"], r1=p["r1"]) for p in laws]
        st["x"], st["y"], st["z"], st["q"] = (torch.cat([p[d] for p in parts]) for d in range(4))
        off = [0]
        for p in laws:
            off.append(off[-1] + p["n"])
        ap = st["ap"] = _context(case)
        ap.build_octree_batched(st["x"], st["y"], st["z"], off)
        ap.stencils()
        ap.deposit(q=st["q"], rtol=st["rtol"], max_iter=MAX_ITER)
        return st
    st["x"], st["y"], st["z"], st["q"] = _particles(case["n"], case["depth"], seed)
    if op == "vp":
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed) + 2)
        v = [torch.randn(case["n"], generator=g, device=DEV, dtype=torch.float64) * 0.01 for _ in range(3)]
        st["vp"] = VlasovPoisson(st["x"], st["y"], st["z"], *v, qm=1.0, rtol=st["rtol"], max_iter=MAX_ITER,
                                 max_depth=case["depth"], c_refine=case["c"], precision=case["precision"],
                                 poly_degree=case["degree"], poly_omega=1.0, device=DEV)
        for ap in st["vp"].ctx:
            ap.set_launch_shape(256, 4, 4, 1)
        return st
    ap = st["ap"] = _context(case)
    if op == "train":
        st["net"] = MPNN(seed=seed, device=DEV)
    if op in ("field", "gather"):
        st["out"] = tuple(torch.empty(case["n"], dtype=torch.float64, device=DEV) for _ in range(4))
    if op in ("operators", "solve", "gather"):
        ap.build_octree(st["x"], st["y"], st["z"])
    if op == "operators":
        st["v"] = _field_vector(ap.n_nodes, seed)
    if op in ("solve", "gather"):
        ap.stencils()
        ap.deposit(q=st["q"], rtol=st["rtol"], max_iter=MAX_ITER)
    if op == "gather":
        # a potential known at the nodes: that of a smoothed unit charge
        r2 = (ap.get_nodes()["xyz"] ** 2).sum(dim=1)
        ap.solve(phi0=-0.0795774715459477 / torch.sqrt(r2 + 0.01), max_iter=0)
    return st


def _field_vector(n, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 3)
    return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)


def run(st):
    case, op = st["case"], st["case"]["op"]
    if op == "vp":
        vp = st["vp"]
        vp.step(1e-4)
        return {"x": vp.x, "y": vp.y, "z": vp.z, "vx": vp.vx, "vy": vp.vy, "vz": vp.vz}
    ap = st["ap"]
    if op in ("solve", "batch"):
        phi, _ = ap.solve(rtol=st["rtol"], max_iter=MAX_ITER)
        return {"phi": phi}
    if op == "operators":
        ap.stencils()
        return {"Av": ap.matvec("A", st["v"]), "Bv": ap.matvec("B", st["v"])}
    if op == "gather":
        phi, ex, ey, ez = ap.gather_field(st["out"])
        return {"phi": phi, "ex": ex, "ey": ey, "ez": ez}
    ap.build_octree(st["x"], st["y"], st["z"])
    if op == "tree":
        return {"leaves": ap.get_leaves(), "nodes": ap.get_nodes()}
    ap.stencils()
    rho, _ = ap.deposit(q=st["q"], rtol=st["rtol"], max_iter=MAX_ITER)
    if op == "train":
        net = st["net"]
        loss = net.loss(ap, backward=True)
        net.adam(ap, 1e-3)
        return {"loss": float(loss["L"]), "grad": net.params()[1]}
    phi, _ = ap.solve(rtol=st["rtol"], max_iter=MAX_ITER)
    field = ap.gather_field(st["out"])
    if case["precision"] == "mixed":
        # the mixed form's particle fields carry FP32 accuracy: kept as FP32
        field = [f.float() for f in field]
    return {"rho": rho, "phi": phi, "phi_p": field[0], "ex": field[1], "ey": field[2], "ez": field[3]}


def work(case):
    """Bytes and FP operations no form of the path can do without: inputs once, outputs once;
    stencils of 24 entries; a solve streams its stored matrix (value and column per entry) once
    per application in the number of Arnoldi steps this method takes at that size."""
    op, beams = case["op"], case.get("beams", 1)
    if op == "batch":   # log-uniform particle counts: their mean, per beam
        n = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
    else:
        n = case["n"]
    each = min(1.35 * (n / case["c"] ** 2) ** 0.6, 8.0 ** case["depth"])   # nodes of a beam
    nodes = beams * each
    mixed, degree = case.get("precision") == "mixed", case.get("degree", 1)
    nnz = 24.0 * nodes
    tree = {"bytes": 24.0 * n + 29.0 * nodes, "flops": 6.0 * n}
    oper = {"bytes": 40.0 * nodes + (9 * 8 + 4 + 16) * nnz, "flops": (450.0 * 24 + 660) * nodes}
    depo = {"bytes": 16.0 * n + 8.0 * nodes, "flops": float(n)}
    gath = {"bytes": 60.0 * n + 8.0 * nodes + (9 * 8 + 4) * nnz, "flops": 38.0 * n + 18.0 * nnz}
    # Arnoldi steps seen: 11 at 1.5e3 nodes to 140 at 1e6 with the degree-16
    # polynomial, 71 at 1.5e3 to 650 at 1.5e4 with Jacobi
    steps = (11.0 if degree > 1 else 70.0) * (each / 1500.0) ** (0.39 if degree > 1 else 0.95)
    entry = (2 + 3) if mixed and degree > 1 else 12
    solv = {"bytes": steps * degree * (entry * nnz + 12.0 * nodes), "flops": steps * degree * 2.0 * nnz}
    parts = {"tree": [tree], "operators": [oper], "solve": [solv], "batch": [solv], "gather": [gath],
             "field": [tree, oper, depo, solv, gath],
             "vp": [tree, oper, depo, solv, gath, {"bytes": 2 * 144.0 * n, "flops": 2 * 12.0 * n}],
             # three layers [2 x 16 | 2 x 64 | 2 x 64] -> 64 forward and twice that backward
             "train": [tree, oper, depo, {"bytes": 16.0 * nnz + 3 * 2.0 * 64 * nodes * 2,
                                          "flops": 3 * 2.0 * (32 + 128 + 128) * 64 * nodes}]}[op]
    return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}


# ---------------------------------------------------------------- 64-bit reference
def exact(case, seed):
    """The method in numpy and torch FP64 for single-beam systems small enough to search in Python."""
    if case["op"] not in ("field", "operators", "solve") or case["n"] > 300_000:
        return None
    if 1.35 * (case["n"] / case["c"] ** 2) ** 0.6 > 14_000 or (case["op"] == "solve" and case["n"] > 2e5):
        return None
    xd, yd, zd, qd = _particles(case["n"], case["depth"], seed)
    pos = torch.stack([xd, yd, zd], dim=1).cpu().numpy()
    q = qd.cpu().numpy()
    depth = case["depth"]
    key = _cell_keys(pos, depth)
    leaf_key, leaf_lev = _leaves(key, depth, case["c"])
    centre, owner, adj = _nodes(leaf_key, leaf_lev, depth)
    n = len(leaf_key)
    nt = len(centre)
    h = 2.0 * 0.5 ** leaf_lev
    row, col, P = _stencils(centre, owner, adj, n)
    lap = P[:, 3] + P[:, 6] + P[:, 8]
    A = torch.zeros(nt, nt, dtype=torch.float64, device=DEV)
    r, c, l = (torch.from_numpy(a).to(DEV) for a in (row, col, lap))
    A.index_put_((r, c), l, accumulate=True)
    diag = torch.zeros(nt, dtype=torch.float64, device=DEV).index_add_(0, r, -l)
    i = torch.arange(nt, device=DEV)
    A[i, i] += diag
    s = torch.zeros(nt, dtype=torch.float64, device=DEV)
    s[:n] = torch.from_numpy(h * h / 24.0).to(DEV)
    B = A * s[:, None]
    B[i, i] += 1.0
    A[i[n:], i[n:]] = 1.0
    if case["op"] == "operators":
        v = _field_vector(nt, seed)
        return {"Av": A @ v, "Bv": B @ v}
    anchor = leaf_key << (3 * (depth - leaf_lev))
    leaf = np.searchsorted(anchor, key, side="right") - 1
    rho_m = np.bincount(leaf, weights=q, minlength=n) / h ** 3
    rho_m = torch.from_numpy(np.concatenate([rho_m, rho_m[owner]])).to(DEV)
    rho = torch.linalg.solve(B, rho_m)
    b = rho.clone()
    b[n:] = 0.0
    phi = torch.linalg.solve(A, b)
    if case["op"] == "solve":
        return {"phi": phi}
    f = phi.cpu().numpy()
    d = np.zeros((n, 9))
    np.add.at(d, row, P * (f[col] - f[row])[:, None])
    dx = pos - (centre[leaf] * 2.0 ** -21 - 1.0)
    g, H = d[leaf, :3], d[leaf][:, [3, 4, 5, 4, 6, 7, 5, 7, 8]].reshape(-1, 3, 3)
    Hd = np.einsum("nij,nj->ni", H, dx)
    E = g + Hd
    return {"rho": rho, "phi": phi, "phi_p": f[leaf] + (g * dx).sum(1) + 0.5 * (dx * Hd).sum(1),
            "ex": E[:, 0], "ey": E[:, 1], "ez": E[:, 2]}


def _spread(v):
    out = np.zeros_like(v)
    for b in range(21):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _morton(c):
    return (_spread(c[:, 0]) << 2) | (_spread(c[:, 1]) << 1) | _spread(c[:, 2])


def _coords(key):
    c = np.zeros((len(key), 3), dtype=np.int64)
    for b in range(21):
        for d in range(3):
            c[:, d] |= ((key >> (3 * b + 2 - d)) & 1) << b
    return c


def _cell_keys(pos, depth):
    c = np.clip(np.floor((pos + 1.0) * 2.0 ** 20), 0, 2 ** 21 - 1).astype(np.int64) >> (21 - depth)
    return _morton(c)


def _leaves(key, depth, c):
    """Keys at their own level and levels of the leaves, in Morton order."""
    opened = [None] * (depth + 1)
    opened[depth] = np.zeros(0, dtype=np.int64)
    for l in range(depth - 1, -1, -1):
        cell, cnt = np.unique(key >> (3 * (depth - l)), return_counts=True)
        want = [cell[cnt * (2.0 * 0.5 ** l) ** 2 >= c * c]]
        up = opened[l + 1]
        if len(up):
            want.append(up >> 3)
            xyz = _coords(up)
            for d in range(3):
                for step in (-1, 1):
                    t = xyz.copy()
                    t[:, d] += step
                    want.append(_morton(t[(t[:, d] >= 0) & (t[:, d] < 2 ** (l + 1))]) >> 3)
        opened[l] = np.unique(np.concatenate(want))
    keys, levs = [], []
    for l in range(depth + 1):
        kids = np.zeros(1, dtype=np.int64) if l == 0 else (opened[l - 1][:, None] * 8 + np.arange(8)).ravel()
        kids = kids[~np.isin(kids, opened[l])]
        keys.append(kids)
        levs.append(np.full(len(kids), l))
    keys, levs = np.concatenate(keys), np.concatenate(levs)
    order = np.argsort(keys << (3 * (depth - levs)), kind="stable")
    return keys[order], levs[order]


def _nodes(key, lev, depth):
    """Integer centres (units of 2^-21) of leaves then boundary nodes, their owners, and the face graph."""
    xyz = _coords(key)
    n = len(key)
    centre = (2 * xyz + 1) << (21 - lev)[:, None]
    index = {(int(l), int(a), int(b), int(c)): i for i, (l, (a, b, c)) in enumerate(zip(lev, xyz))}
    adj = [[] for _ in range(n)]
    extra, owner = [], []
    for face in range(6):
        d, up = face >> 1, face & 1
        for j in range(n):
            l = int(lev[j])
            t = [int(v) for v in xyz[j]]
            t[d] += 1 if up else -1
            if t[d] < 0 or t[d] >= 1 << l:
                p = centre[j].copy()
                p[d] = (1 << 22) if up else 0
                adj[j].append(n + len(extra))
                extra.append(p)
                owner.append(j)
                continue
            k = index.get((l, *t))
            if k is None:
                k = index.get((l - 1, *(v >> 1 for v in t)))
            if k is not None:
                adj[j].append(k)
                continue
            for o in range(4):
                kid = [2 * v for v in t]
                rest = [e for e in range(3) if e != d]
                kid[d] += 0 if up else 1
                kid[rest[0]] += o >> 1
                kid[rest[1]] += o & 1
                adj[j].append(index[(l + 1, *kid)])
    owner = np.array(owner, dtype=np.int64)
    return np.concatenate([centre, np.array(extra, dtype=np.int64).reshape(-1, 3)]), owner, adj


def _select(cand, d2, oct_, m_target):
    """Positions, in (distance, index) order, of the octant picks, the nearest fill and its ties."""
    seen = [0] * 8
    pick = np.zeros(len(cand), dtype=bool)
    for p, o in enumerate(oct_):
        if seen[o] < 2:
            seen[o] += 1
            pick[p] = True
    rest = np.flatnonzero(~pick)
    need = max(0, m_target - int(pick.sum()))
    fill = rest[:need]
    room = 32 - int(pick.sum()) - need
    if need and len(fill) == need:
        tie = rest[need:]
        fill = np.concatenate([fill, tie[d2[tie] == d2[fill[-1]]][:max(0, room)]])
    pick[fill] = True
    return np.flatnonzero(pick)


def _wls(off):
    """9 x m operator of one stencil, or None where it is not usable."""
    hmax = np.abs(off).max()
    xi = off / hmax
    r2 = (off.astype(np.float64) ** 2).sum(1)
    w = (np.exp(-r2 / r2.max()) - math.exp(-4)) / (1 - math.exp(-4))
    x, y, z = xi.T
    V = np.stack([x, y, z, x * x / 2, x * y, x * z, y * y / 2, y * z, z * z / 2], axis=1) * w[:, None]
    Q, R = np.linalg.qr(V)
    d = np.abs(np.diag(R))
    if len(off) < 9 or d.min() < 1e-6 * d.max():
        return None
    P = np.linalg.solve(R, Q.T) * w
    h = hmax * 2.0 ** -21
    P[:3] /= h
    P[3:] /= h * h
    return P if (P[3] + P[6] + P[8]).sum() > 0 else None


def _stencils(centre, owner, adj, n):
    """Row, column and the nine derivative weights of every stencil entry."""
    rows, cols, ops = [], [], []
    for j in range(n):
        ring, front, found = [j], [j], None
        seen = {j}
        for k in range(1, 6):
            new = []
            for u in front:
                for v in (adj[u] if u < n else (int(owner[u - n]),)):
                    if v not in seen:
                        seen.add(v)
                        new.append(v)
            ring += new
            front = new
            if k < 2 or len(ring) - 1 < (20 if k < 5 else 9):
                continue
            cand = np.array(ring[1:], dtype=np.int64)
            off = centre[cand] - centre[j]
            d2 = (off * off).sum(1)
            order = np.lexsort((cand, d2))
            cand, off, d2 = cand[order], off[order], d2[order]
            oct_ = ((off >= 0) * np.array([4, 2, 1])).sum(1)
            for m_target in range(20, 33, 2):
                s = _select(cand, d2, oct_, m_target)
                P = _wls(off[s])
                if P is not None:
                    found = (cand[s], P)
                if P is not None or len(s) >= len(cand):
                    break
            if found:
                break
        rows.append(np.full(len(found[0]), j, dtype=np.int64))
        cols.append(found[0])
        ops.append(found[1].T)
    return np.concatenate(rows), np.concatenate(cols), np.concatenate(ops)
