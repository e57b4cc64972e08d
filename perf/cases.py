"""What the framework is timed on: the calls its users make, through the Python binding.

A case is one kind of call at one size:

  step    a triangulation that is kept while points move: a pass is a few time steps (one
          kdt_step each, a move list per step) and the export of the triangle list that a
          simulation reads after them
  batch   the same for many independent instances in one handle
  build   the triangulation of a new point set, and its export
  dvals   the N-th nearest-neighbour distances of every point (d-calculation)
  infer   the proposal network on the rows of a step's moves
  train   one optimiser step of the proposal network: loss, gradient, Adam

The sizes are those of the repository's own workloads (paper_2308_06484_gb300.workloads):
1e3 to 16e6 points, 1 to 16 moves per partition, moves of one unit up to several point
spacings, 1 to 512 instances.  Points and moves are drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2308_06484_gb300 import kdt, proposal

DEV = "cuda"
SHAPES = ((64, 32), (64,), (64, 64), (64,), (18, 64), (18,))  # the network's parameters, one flat array
PARAMS = 7442


def listed():
    return [
        # the smallest workload (c1): 16 one-unit moves a step from host memory; latency
        {"name": "step_small", "kind": "step", "n": 1000, "bits": 16, "points": "uniform", "grid": 4, "mpc": 1,
         "dist": 1, "steps": 8, "moves": "host", "variant": 0, "learned": False},
        # the ordinary one (c2): a million uniform points, one short move per partition
        {"name": "step_uniform", "kind": "step", "n": 1000000, "bits": 24, "points": "uniform", "grid": 64, "mpc": 1,
         "dist": 8, "steps": 8, "moves": "device", "variant": 0, "learned": False},
        # the largest one (c3): 32 Gaussians and 5 % lattice (cocircular points), 1-16
        # moves per partition: about half a million moves a pass
        {"name": "step_clustered", "kind": "step", "n": 16000000, "bits": 24, "points": "clustered", "grid": 256,
         "mpc": 16, "dist": 8, "steps": 4, "moves": "device", "variant": 0, "learned": False},
        # points that jump: moves of up to about two point spacings, which leave the star
        {"name": "step_far", "kind": "step", "n": 200000, "bits": 24, "points": "uniform", "grid": 28, "mpc": 4,
         "dist": 80000, "steps": 8, "moves": "device", "variant": 0, "learned": False},
        # the ordinary one with the trained proposal, evaluated by the step planner (c5)
        {"name": "step_learned", "kind": "step", "n": 1000000, "bits": 24, "points": "uniform", "grid": 64, "mpc": 1,
         "dist": 8, "steps": 8, "moves": "device", "variant": 0, "learned": True},
        # 512 instances of 1e3 to 2e5 points advanced together (c4)
        {"name": "step_batch", "kind": "batch", "instances": 512, "lo": 1000, "hi": 200000, "mpc": 4, "dist": 8,
         "steps": 4},
        # the build every use starts from (and the full rebuild a step is compared with)
        {"name": "build_uniform", "kind": "build", "n": 1000000, "bits": 24, "points": "uniform", "instances": 1},
        # many small sets built at once
        {"name": "build_batch", "kind": "build", "n": 1500000, "bits": 20, "points": "uniform", "instances": 128},
        # the paper's d-calculation, with the partition minima
        {"name": "dvals", "kind": "dvals", "n": 1000000, "bits": 24, "points": "uniform", "N": 4},
        # the network on the moves of one step of the largest workload
        {"name": "infer", "kind": "infer", "rows": 165000},
        # one training step on a mini-batch (rows picked by index), as the trainer takes it
        {"name": "train_batch", "kind": "train", "rows": 8192, "pool": 480000, "index": True},
        # the gradient over a whole trace
        {"name": "train_full", "kind": "train", "rows": 262144, "pool": 262144, "index": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "build", "build", "dvals", "infer", "train"])
    if kind == "step":
        n = _log(rng, 300, 4000000)
        bits = rng.choice([b for b in (16, 20, 24, 28) if (1 << (2 * b)) >= 1024 * n])
        spacing = (1 << bits) / math.sqrt(n)
        return {"kind": kind, "n": n, "bits": bits, "points": rng.choice(["uniform", "clustered"]),
                "grid": max(1, int(round(math.sqrt(n / rng.uniform(100.0, 500.0))))), "mpc": rng.choice([1, 1, 4, 16]),
                "dist": rng.choice([1, 8, 8, max(8, int(spacing * rng.uniform(0.1, 2.0)))]),
                "steps": rng.choice([2, 4, 8]), "moves": rng.choice(["host", "device", "device"]),
                "variant": rng.choice([0, 0, 0, 0, 1, 2]), "learned": rng.random() < 0.1}
    if kind == "batch":
        hi = _log(rng, 2000, 200000)
        return {"kind": kind, "instances": _log(rng, 2, 256), "lo": rng.choice([300, 1000]), "hi": hi,
                "mpc": rng.choice([1, 4]), "dist": rng.choice([1, 8, 64]), "steps": rng.choice([2, 4])}
    if kind == "build":
        inst = rng.choice([1, 1, 1, _log(rng, 2, 300)])
        n = _log(rng, 300, 4000000) if inst == 1 else _log(rng, 400 * inst, max(500 * inst, 2000000))
        bits = rng.choice([b for b in (16, 20, 24, 28) if (1 << (2 * b)) >= 1024 * n])
        return {"kind": kind, "n": n, "bits": bits, "points": rng.choice(["uniform", "clustered"]) if inst == 1
                else "uniform", "instances": inst}
    if kind == "dvals":
        return {"kind": kind, "n": _log(rng, 300, 4000000), "bits": 24, "points": rng.choice(["uniform", "clustered"]),
                "N": rng.choice([1, 2, 4, 9])}
    if kind == "infer":
        return {"kind": kind, "rows": _log(rng, 100, 1000000)}
    rows = _log(rng, 200, 500000)
    return {"kind": kind, "rows": rows, "pool": rows + rng.randrange(0, 100000), "index": True}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1000003 + 17)
    return g


def _key(p):
    return (p[..., 0] << 32) | p[..., 1]


def _first_of(keys):
    """Positions of the first occurrence of every key, in increasing position order."""
    s, order = torch.sort(keys, stable=True)
    new = torch.ones_like(s, dtype=torch.bool)
    new[1:] = s[1:] != s[:-1]
    return torch.sort(order[new])[0]


def _points(g, n, bits, shape):
    """n distinct points (int64, n x 2): uniform, or 32 Gaussians with 5 % square lattice."""
    L = 1 << bits
    have = torch.empty((0, 2), dtype=torch.int64, device=DEV)
    if shape == "clustered":
        centres = torch.rand((32, 2), generator=g, device=DEV, dtype=torch.float64) * L
        n_lat = int(round(0.05 * n))
        side = max(1, int(math.ceil(math.sqrt(n_lat / 8.0))))
        step = max(1, min(64, L // (4 * side)))
        a = torch.arange(side, device=DEV, dtype=torch.int64) * step
        # eight patches, each inside one of the clusters
        o = centres[:8] + torch.randn((8, 2), generator=g, device=DEV, dtype=torch.float64) * (L / 128.0)
        o = o.to(torch.int64).clamp(0, L - 1 - (side - 1) * step)
        lat = (torch.stack(torch.meshgrid(a, a, indexing="ij"), -1)[None] + o[:, None, None]).reshape(-1, 2)[:n_lat]
        have = lat[_first_of(_key(lat))]
    while have.shape[0] < n:
        m = (n - have.shape[0]) * 17 // 16 + 64
        if shape == "uniform":
            c = torch.randint(0, L, (m, 2), generator=g, device=DEV)
        else:
            k = torch.randint(0, 32, (m,), generator=g, device=DEV)
            c = centres[k] + torch.randn((m, 2), generator=g, device=DEV, dtype=torch.float64) * (L / 64.0)
            c = torch.round(c).to(torch.int64)
            c = c[((c >= 0) & (c < L)).all(1)]
        have = torch.cat([have, c])
        have = have[_first_of(_key(have))]
    have = have[:n]
    return have[torch.randperm(n, generator=g, device=DEV)].contiguous()


def _subsets(g, cells, ncell, mpc, k):
    """k disjoint sets of point ids, each with 1 to mpc random points of every cell (as far as
    the cell has them): one list of ids per set, ordered by cell."""
    n = cells.shape[0]
    order = torch.randperm(n, generator=g, device=DEV)
    order = order[torch.sort(cells[order], stable=True)[1]]
    c = cells[order]
    counts = torch.bincount(c, minlength=ncell)
    rank = torch.arange(n, device=DEV) - (torch.cumsum(counts, 0) - counts)[c]
    lo = torch.zeros(ncell, dtype=torch.int64, device=DEV)
    sets = []
    for _ in range(k):
        hi = lo + torch.randint(1, mpc + 1, (ncell,), generator=g, device=DEV)
        sets.append(order[(rank >= lo[c]) & (rank < hi[c])])
        lo = hi
    return sets


def _moves(g, pos, x0, bits, cells, ncell, case):
    """The move lists of a pass: half of its steps move one set of points each to a place
    A, the other half move the same sets on to a place B, every move along an axis by 1 to
    dist units.  All places are distinct and free, so a pass can be repeated (B, A, B) and
    always ends in the same positions.  x0: where a point's instance begins in x."""
    L = 1 << bits
    dirs = torch.tensor([[1, 0], [-1, 0], [0, 1], [0, -1]], device=DEV)
    sets = _subsets(g, cells, ncell, case["mpc"], case["steps"] // 2)
    ids = torch.cat(sets)
    own = torch.cat([torch.full_like(s, i) for i, s in enumerate(sets)])

    def hop(p):
        d = torch.randint(0, 4, (p.shape[0],), generator=g, device=DEV)
        s = torch.randint(1, case["dist"] + 1, (p.shape[0], 1), generator=g, device=DEV)
        return p + dirs[d] * s

    a = hop(pos[ids])
    b = hop(a)
    # inside the domain, distinct from every position and from every other target
    m, n = ids.shape[0], pos.shape[0]
    first = torch.zeros(n + 2 * m, dtype=torch.bool, device=DEV)
    first[_first_of(_key(torch.cat([pos, a, b])))] = True
    ok = first[n:n + m] & first[n + m:]
    for t in (a, b):
        x = t[:, 0] - x0[ids]
        ok &= (x >= 0) & (x < L) & (t[:, 1] >= 0) & (t[:, 1] < L)
    out = []
    for to in (a, b):
        for i in range(len(sets)):
            sel = ok & (own == i)
            out.append((ids[sel], to[sel]))
    return out


def _cells(pos, grid, bits):
    return ((pos[:, 1] * grid) >> bits) * grid + ((pos[:, 0] * grid) >> bits)


def _rows(g, rows):
    """Rows like those a trace holds: a short move, a degree, link vertices about one mean
    radius away; slots and cavity sizes."""
    x = torch.randn((rows, 32), generator=g, device=DEV) * 0.7
    x[:, 0] = torch.rand(rows, generator=g, device=DEV) * 0.05
    k = torch.randint(4, 10, (rows,), generator=g, device=DEV)
    x[:, 1] = k / 16.0
    x[:, 2:] *= (torch.arange(15, device=DEV)[None] < k[:, None]).repeat_interleave(2, 1)
    slot = torch.randint(0, 6, (rows,), generator=g, device=DEV) + (torch.rand(rows, generator=g, device=DEV) < 0.1) * 10
    y = torch.stack([slot, k - 2], 1).to(torch.int32)
    return x.contiguous(), y.contiguous()


def _network(g):
    """He-uniform weights and small biases: FP32 masters and their BF16 rounding."""
    parts = []
    for shape in SHAPES:
        lim = math.sqrt(6.0 / shape[1]) if len(shape) == 2 else 0.1
        parts.append(((torch.rand(shape, generator=g, device=DEV) * 2 - 1) * lim).reshape(-1))
    master = torch.cat(parts)
    return master, master.to(torch.bfloat16).view(torch.int16).contiguous()


def _infer_inputs(case, seed):
    g = _gen(seed)
    return {"x": _rows(g, case["rows"])[0], "params": _network(g)[1]}


def _train_inputs(case, seed):
    g = _gen(seed)
    x, y = _rows(g, case["pool"])
    master, params = _network(g)
    index = torch.randperm(case["pool"], generator=g, device=DEV)[:case["rows"]].contiguous() if case["index"] else None
    # moments as in the middle of a training run
    m = torch.randn(PARAMS, generator=g, device=DEV) * 1e-2
    v = torch.rand(PARAMS, generator=g, device=DEV) * 1e-3 + 1e-4
    return {"x": x, "y": y, "index": index, "master": master, "params": params, "m": m, "v": v, "t": 50}


# ---------------------------------------------------------------- prepare / run

def _triangles(n):
    """Room for the triangle list of n points (at most 2n - 5 rows; the rest stays zero)."""
    return torch.zeros((2 * n, 3), dtype=torch.int32, device=DEV)


def _exported(s):
    rows = s["tri"].export_triangles(s["out"]).shape[0]
    return {"triangles": s["out"], "rows": rows}


def _prepare_step(case, g):
    n, bits, grid = case["n"], case["bits"], case["grid"]
    pos = _points(g, n, bits, case["points"])
    lists = _moves(g, pos, torch.zeros_like(pos[:, 0]), bits, _cells(pos, grid, bits), grid * grid, case)
    moves = [torch.cat([i[:, None], t], 1).to(torch.int32).contiguous() for i, t in lists]
    if case["moves"] == "host":
        moves = [m.cpu().numpy() for m in moves]
    tri = kdt.Triangulation(kdt.default_config(grid=grid, domain_bits=bits, variant=case["variant"],
                                               plan=6 if case["learned"] else 0))
    tri.build(pos.to(torch.int32).contiguous())
    if case["learned"]:  # a short training on the rows of the first steps
        tr = proposal.Trace(sum(len(m) for m in moves))
        tr.attach(tri)
        for m in moves:
            tri.step(m)
        tr.detach(tri)
        x, y = tr.view()
        tn = proposal.Trainer(tri, seed=0, tensor_cores=True)
        tn.fit(x, y, epochs=4, batch=1024)
        tri.set_proposal(tn.params)
    return {"tri": tri, "moves": moves, "out": _triangles(n)}


def _sizes(case):
    g = _gen(case["instances"])  # the same sizes for every seed
    lo, hi = math.log(case["lo"]), math.log(max(case["hi"], case["lo"] + 1))
    return torch.floor(torch.exp(lo + torch.rand(case["instances"], generator=g, device=DEV, dtype=torch.float64)
                                 * (hi - lo))).to(torch.int64)


def _instances(g, sizes, bits):
    """Distinct uniform points of every instance (no two of one instance alike), back to back."""
    inst = torch.repeat_interleave(torch.arange(sizes.shape[0], device=DEV), sizes)
    pos = torch.randint(0, 1 << bits, (inst.shape[0], 2), generator=g, device=DEV)
    while True:  # redraw the few that coincide
        keys = _key(pos) ^ (inst << 52)
        again = torch.ones(inst.shape[0], dtype=torch.bool, device=DEV)
        again[_first_of(keys)] = False
        k = int(again.sum())
        if k == 0:
            return pos, inst
        pos[again] = torch.randint(0, 1 << bits, (k, 2), generator=g, device=DEV)


def _split(pos, sizes):
    return list(np.split(pos.to(torch.int32).cpu().numpy(), np.cumsum(sizes.cpu().numpy())[:-1]))


def _prepare_batch(case, g):
    bits = 20
    sizes = _sizes(case)
    pos, inst = _instances(g, sizes, bits)
    side = torch.clamp(torch.round(torch.sqrt(sizes.double() / 256.0)).to(torch.int64), min=1)
    first_cell = torch.cumsum(side * side, 0) - side * side
    G = side[inst]
    cells = first_cell[inst] + ((pos[:, 1] * G) >> bits) * G + ((pos[:, 0] * G) >> bits)
    start = torch.cumsum(sizes, 0) - sizes
    # every instance in a band of its own in x while targets are compared
    x0 = inst << (bits + 1)
    band = pos.clone()
    band[:, 0] += x0
    moves, offs = [], []
    for ids, to in _moves(g, band, x0, bits, cells, int((side * side).sum()), case):
        local = torch.stack([ids - start[inst[ids]], to[:, 0] - x0[ids], to[:, 1]], 1)
        moves.append(local.to(torch.int32).contiguous())
        cnt = torch.bincount(inst[ids], minlength=sizes.shape[0]).cpu().numpy()
        offs.append(np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64))
    tri = kdt.Triangulation(kdt.default_config(domain_bits=bits))
    tri.build_batch(_split(pos, sizes))
    return {"tri": tri, "moves": moves, "offs": offs,
            "out": _triangles(pos.shape[0])}


def _prepare_build(case, g):
    n, bits = case["n"], case["bits"]
    tri = kdt.Triangulation(kdt.default_config(domain_bits=bits))
    out = _triangles(n)
    if case["instances"] == 1:
        return {"tri": tri, "xy": _points(g, n, bits, case["points"]).to(torch.int32).contiguous(), "out": out}
    w = torch.exp(torch.rand(case["instances"], generator=_gen(case["instances"]), device=DEV, dtype=torch.float64) * 3.0)
    sizes = torch.clamp((w / w.sum() * n).to(torch.int64), min=16)
    pos, _ = _instances(g, sizes, bits)
    return {"tri": tri, "xys": _split(pos, sizes),
            "out": _triangles(pos.shape[0])}


def _prepare_dvals(case, g):
    n = case["n"]
    tri = kdt.Triangulation(kdt.default_config(domain_bits=case["bits"]))
    tri.build(_points(g, n, case["bits"], case["points"]).to(torch.int32).contiguous())
    return {"tri": tri, "N": case["N"], "dist2": torch.empty(n, dtype=torch.int64, device=DEV),
            "cmin": torch.empty(tri.num_cells(), dtype=torch.int64, device=DEV)}


def _prepare_infer(case, seed):
    s = _infer_inputs(case, seed)
    s["tri"] = kdt.Triangulation(kdt.default_config())
    s["out"] = torch.empty((case["rows"], 18), dtype=torch.float32, device=DEV)
    return s


def _prepare_train(case, seed):
    s = _train_inputs(case, seed)
    s["tri"] = kdt.Triangulation(kdt.default_config())
    s["grad"], s["loss"] = torch.zeros(PARAMS, device=DEV), torch.zeros(1, device=DEV)
    return s


def prepare(case, seed):
    g = _gen(seed)
    k = case["kind"]
    s = (_prepare_step(case, g) if k == "step" else _prepare_batch(case, g) if k == "batch"
         else _prepare_build(case, g) if k == "build" else _prepare_dvals(case, g) if k == "dvals"
         else _prepare_infer(case, seed) if k == "infer" else _prepare_train(case, seed))
    s["kind"] = k
    return s


def run(s):
    tri, k = s["tri"], s["kind"]
    if k == "step":
        for mv in s["moves"]:
            tri.step(mv)
        return _exported(s)
    if k == "batch":
        for mv, offs in zip(s["moves"], s["offs"]):
            tri.step_batch(mv, offs)
        return _exported(s)
    if k == "build":
        if "xy" in s:
            tri.build(s["xy"])
        else:
            tri.build_batch(s["xys"])
        return _exported(s)
    if k == "dvals":
        info = tri.d_values(s["N"], s["dist2"], s["cmin"])
        return {"dist2": s["dist2"], "cell_min2": s["cmin"], "min2": info["min2"], "max_degree": info["max_degree"]}
    if k == "infer":
        tri.mlp_forward_tc(s["params"], s["x"], s["out"])
        return s["out"]
    tri.mlp_loss_grad(s["params"], s["x"], s["y"], s["grad"], s["loss"], index=s["index"], tensor_cores=True)
    s["t"] += 1
    tri.mlp_adam(s["master"], s["grad"], s["m"], s["v"], s["t"], 2e-3, params_bf16=s["params"])
    return {"grad": s["grad"], "loss": s["loss"], "master": s["master"], "m": s["m"], "v": s["v"]}


# ---------------------------------------------------------------- what a pass needs

def work(case):
    """A moved point: its old and its new star read and written once (688 bytes at the mean
    degree 6: 32 + 16 per triangle, 8 per vertex) and the move itself; an export: the
    vertices of 2n triangles read, the list written; a build: the points read, 2n triangles
    of 32 bytes written; the network: its rows and outputs, its products."""
    k = case["kind"]
    if k == "step":
        cells = case["grid"] ** 2 * (0.45 if case["points"] == "clustered" else 1.0)
        m = min(case["n"] / 2.0, cells * (1 + case["mpc"]) / 2.0) * case["steps"]
        return {"bytes": m * 700 + 2 * case["n"] * 28, "flops": 0}
    if k == "batch":
        n = case["instances"] * (case["hi"] - case["lo"]) / max(1e-9, math.log(max(case["hi"], case["lo"] + 1)
                                                                           / case["lo"]))
        return {"bytes": n / 256.0 * (1 + case["mpc"]) / 2.0 * case["steps"] * 700 + 2 * n * 28, "flops": 0}
    if k == "build":
        return {"bytes": case["n"] * (8 + 64 + 56), "flops": 0}
    if k == "dvals":
        return {"bytes": case["n"] * (2 * 12 + 8 + 8), "flops": 0}
    if k == "infer":
        return {"bytes": case["rows"] * (32 + 18) * 4, "flops": case["rows"] * 2 * 7296}
    return {"bytes": case["rows"] * (34 * 4 + (8 if case["index"] else 0)) + 7442 * 4 * 8,
            "flops": case["rows"] * 2 * (2 * 7296 + 18 * 64 + 64 * 64)}


# ---------------------------------------------------------------- the same in 64 bits

def _forward64(p, x):
    o = 0
    w = []
    for s in SHAPES:
        k = math.prod(s)
        w.append(p[o:o + k].view(s))
        o += k
    h = torch.relu(x @ w[0].T + w[1])
    h = torch.relu(h @ w[2].T + w[3])
    return h @ w[4].T + w[5]


def exact(case, seed):
    k = case["kind"]
    if k not in ("infer", "train"):
        return None  # whole numbers
    s = (_infer_inputs if k == "infer" else _train_inputs)(case, seed)
    p = s["params"].view(torch.bfloat16).double().requires_grad_(k == "train")
    if k == "infer":
        return torch.cat([_forward64(p, x.double()) for x in s["x"].split(100000)])
    x, y = (s["x"], s["y"]) if s["index"] is None else (s["x"][s["index"]], s["y"][s["index"]])
    grad, loss = torch.zeros_like(p), 0.0
    for xs, ys in zip(x.split(100000), y.split(100000)):
        out = _forward64(p, xs.double())
        part = (torch.nn.functional.cross_entropy(out[:, :17], ys[:, 0].long(), reduction="sum")
                + 0.25 * (out[:, 17] - torch.log2(ys[:, 1].double())).square().sum()) / x.shape[0]
        grad += torch.autograd.grad(part, p)[0]
        loss += float(part.detach())
    t, b1, b2 = s["t"] + 1, 0.9, 0.999
    m = b1 * s["m"].double() + (1 - b1) * grad
    v = b2 * s["v"].double() + (1 - b2) * grad * grad
    master = s["master"].double() - 2e-3 * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + 1e-8)
    return {"grad": grad, "loss": torch.tensor([loss], dtype=torch.float64), "master": master, "m": m, "v": v}
