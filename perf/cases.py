"""What the library is timed on: batches, products, reads and training through its public entry points.

A *pass* is what a program does each time new updates arrive.  A long-running program keeps its handle and its
page-locked result arrays and applies one batch after the other, so each dynamic case keeps a short ring of batches in
which every batch is followed by the one that undoes it: the matrix stays the size it was, however often the pass is
repeated, and the handle has already taken a few batches when the pass begins, as it has in such a program.
"""

import math
import random
import zlib
from types import SimpleNamespace

import numpy as np
import torch

import paper_2202_08808_gb300 as dspg

F64, I32 = dspg.PLUS_TIMES_F64, dspg.MIN_PLUS_I32
GRAPH500 = (0.57, 0.19, 0.19, 0.05)
FLAT = (0.45, 0.15, 0.15, 0.25)
INS, DEL, SET = dspg.OP_INSERT, dspg.OP_DELETE, dspg.OP_SET
PAIRS = 3   # batches of a ring, each with the one that undoes it
WARM = 4    # passes the handle has taken before


def listed():
    return [
        # a small general sparse product kept current, the whole of C read back after each batch
        {"name": "er-4096-1024", "family": "er", "n": 4096, "k": 4096, "m": 4096, "per_row": 8, "both": False,
         "semiring": F64, "updates": 1024},
        # a trickle of changes to a mesh operator: the latency of one small batch and the read of its rows
        {"name": "stencil-64-16", "family": "stencil", "nx": 64, "ny": 64, "nz": 64, "updates": 16, "device": False},
        # the mesh operator at its usual batch, 0.07 % of the entries
        {"name": "stencil-128-1e4", "family": "stencil", "nx": 128, "ny": 128, "nz": 128, "updates": 10000,
         "device": False},
        # the same with a large batch, where a quarter of the rows change
        {"name": "stencil-128-1e5", "family": "stencil", "nx": 128, "ny": 128, "nz": 128, "updates": 100000,
         "device": True},
        # multi-source path relaxation on a skewed graph: few, wide rows of C, hubs of A
        {"name": "paths-20-1000", "family": "paths", "scale": 20, "cols": 256, "edges": 1000, "device": True},
        # the square of a skewed graph: rows of C of every length, most of them long
        {"name": "square-18-300", "family": "square", "scale": 18, "semiring": F64, "edges": 300, "sizing": "bound",
         "bloom": False},
        # the same kind of graph kept by the entry-level masked recompute
        {"name": "masked-17-1000", "family": "square", "scale": 17, "semiring": F64, "edges": 1000,
         "sizing": "bound", "bloom": True},
        # a sliding window over a mesh: a batch of insertions by the delta path, and its expiry by the row path
        {"name": "window-96-5000", "family": "window", "nx": 96, "ny": 96, "nz": 96, "updates": 5000},
        # uneven instances of both semirings, one batch each, in one group
        {"name": "group-12", "family": "group", "members": 12, "lo": 10, "hi": 13, "updates": 1000},
        # the full product of the mesh operator, computed afresh and read on the device
        {"name": "static-128", "family": "static", "nx": 128, "ny": 128, "nz": 128},
        # a handle built for a skewed graph, read and closed: what a program pays at its start
        {"name": "build-15", "family": "build", "scale": 15, "semiring": F64},
        # the row-size estimator trained on rows the library produced
        {"name": "train-4096", "family": "estimator", "op": "train", "scale": 15, "batch": 4096, "steps": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["er", "stencil", "stencil", "paths", "square", "square", "window", "group", "static", "build",
                    "estimator"])
    if f == "er":
        n, both = _log(rng, 500, 20000), rng.random() < 0.5
        k, m = (_log(rng, 500, 20000), _log(rng, 1100, 20000)) if both else (n, n)
        return {"family": f, "n": n, "k": k, "m": m, "per_row": rng.randint(3, 12), "both": both,
                "semiring": rng.choice([F64, I32]), "updates": _log(rng, 8, n / 4)}
    if f in ("stencil", "window", "static"):
        hi = {"stencil": 128, "window": 96, "static": 128}[f]
        d = {"family": f, "nx": _log(rng, 20, hi), "ny": _log(rng, 20, hi), "nz": _log(rng, 20, hi)}
        n = d["nx"] * d["ny"] * d["nz"]
        if f != "static":
            d["updates"] = _log(rng, 1, n / 20) if f == "stencil" else _log(rng, 10, n / 100)
        if f == "stencil":
            d["device"] = rng.random() < 0.5
        return d
    if f == "paths":
        scale = rng.randint(14, 20)
        return {"family": f, "scale": scale, "cols": _log(rng, 30, 900), "edges": _log(rng, 10, 2 ** (scale - 9)),
                "device": rng.random() < 0.5}
    if f == "square":
        bloom = rng.random() < 0.4
        scale = rng.randint(12, 17)
        return {"family": f, "scale": scale, "semiring": rng.choice([F64, I32]),
                "edges": _log(rng, 10, 2 ** (scale - 9)),
                "sizing": "bound" if bloom else rng.choice(["bound", "bound", "learned", "exact"]), "bloom": bloom}
    if f == "group":
        lo = rng.randint(9, 11)
        return {"family": f, "members": rng.randint(3, 12), "lo": lo, "hi": lo + rng.randint(0, 2),
                "updates": _log(rng, 10, 1000)}
    if f == "build":
        return {"family": f, "scale": rng.randint(10, 15), "semiring": rng.choice([F64, I32])}
    return {"family": f, "op": rng.choice(["train", "grad", "predict"]), "scale": rng.randint(13, 15),
            "batch": _log(rng, 500, 8192), "steps": rng.randint(8, 32)}


# ----------------------------------------------------------------- inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Draw:
    """Random numbers of a stream of its own."""

    def __init__(self, seed):
        self.g = torch.Generator(device=_device())
        self.g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 17)

    def uniform(self, n):
        return torch.rand(n, generator=self.g, device=_device(), dtype=torch.float64)

    def below(self, n, hi):
        return torch.randint(0, hi, (n,), generator=self.g, device=_device(), dtype=torch.int64)

    def order(self, n):
        return torch.randperm(n, generator=self.g, device=_device())

    def values(self, n, sr):
        return self.uniform(n) if sr == F64 else (1 + self.below(n, 100)).to(torch.int32)

    def mesh_values(self, n):
        return -1.0 + 0.2 * (self.uniform(n) - 0.5)


def _shape_of(case):
    """The stream that a case's structure is drawn from.  The same for every seed: a seed renames the vertices and draws
    the values, so that results of other seeds have other places and other numbers, but the same sizes."""
    plain = sorted((k, v) for k, v in case.items() if k != "name")
    return _Draw(zlib.crc32(repr(plain).encode()))


def _parts(key, ncols):
    row = torch.div(key, ncols, rounding_mode="floor")
    return row, key - row * ncols


class Mat:
    """A canonical CSR on the device: `key` = row * ncols + column ascending, with the arrays a handle is built from."""

    def __init__(self, nrows, ncols, key, val):
        self.nrows, self.ncols, self.key, self.val = nrows, ncols, key, val
        self.rows, col = _parts(key, ncols)
        self.col = col.to(torch.int32)
        self.rowptr = torch.zeros(nrows + 1, dtype=torch.int64, device=key.device)
        self.rowptr[1:] = torch.cumsum(torch.bincount(self.rows, minlength=nrows), 0)


def _updates(key, val, op, ncols):
    row, col = _parts(key, ncols)
    return SimpleNamespace(row=row.to(torch.int32), col=col.to(torch.int32), val=val, op=op, key=key)


def _undo(A, b):
    """The batch that takes A with b applied back to A."""
    key = torch.unique(b.key)
    at = torch.searchsorted(A.key, key).clamp(max=A.key.numel() - 1)
    there = A.key[at] == key
    op = torch.where(there, torch.full_like(key, SET), torch.full_like(key, DEL)).to(torch.uint8)
    return _updates(key, torch.where(there, A.val[at], torch.zeros_like(A.val[:1])), op, A.ncols)


def _ring(A, batches):
    return [x for b in batches for x in (b, _undo(A, b))]


def _on_host(b):
    """The batch in page-locked host memory, as it comes in from outside."""
    def pin(t):
        return t.cpu().pin_memory().numpy() if torch.cuda.is_available() else t.cpu().numpy()
    return SimpleNamespace(row=pin(b.row), col=pin(b.col), val=pin(b.val), op=pin(b.op))


def _mixed(shape, d, key, val, ncols):
    """A third each of insertions, deletions and value changes, in random order, at the given positions."""
    op = (shape.order(key.numel()) % 3).to(torch.uint8)
    return _updates(key, torch.where(op == DEL, torch.zeros_like(val[:1]), val), op, ncols)


def _scattered(case, shape, d):
    """A (and B) with rows of about per_row distinct uniform columns, and mixed batches, half at present entries."""
    sr, n, k, m = case["semiring"], case["n"], case["k"], case["m"]
    names = [d.order(x) for x in (n, k, m)]
    if not case["both"]:
        names = [names[0]] * 3

    def one(rows, cols, by_row, by_col, count):
        r = torch.arange(rows, device=_device()).repeat_interleave(case["per_row"])
        raw = torch.unique(r * cols + shape.below(rows * case["per_row"], cols))

        def named(key):
            i, j = _parts(key, cols)
            return by_row[i] * cols + by_col[j]

        M = Mat(rows, cols, torch.sort(named(raw)).values, d.values(raw.numel(), sr))
        batches = []
        for _ in range(PAIRS):
            key = torch.where(shape.uniform(count) < 0.5, raw[shape.below(count, raw.numel())], shape.below(count, rows * cols))
            batches.append(_mixed(shape, d, named(key), d.values(count, sr), cols))
        return M, _ring(M, batches)

    A, ring = one(n, k, names[0], names[1], case["updates"])
    B, ring_b = one(k, m, names[1], names[2], max(1, case["updates"] // 8)) if case["both"] else (None, None)
    return sr, A, B, ring, ring_b


def _mesh(case, shape, d):
    """The 7-point operator of an nx x ny x nz grid (diagonal 6, neighbours -1 + U(-0.1, 0.1)) and batches at positions
    (i, j) with j within two grid hops of i: mixed ones, or for a window insertions two hops away."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    flip = [bool(x) for x in d.below(3, 2).tolist()]

    def at(x, y, z):
        x, y, z = ((s - 1 - c if on else c) for c, s, on in zip((x, y, z), (nx, ny, nz), flip))
        return x + nx * (y + ny * z)

    def xyz(i):
        return i % nx, torch.div(i, nx, rounding_mode="floor") % ny, torch.div(i, nx * ny, rounding_mode="floor")

    def pairs(i, dx, dy, dz):
        x, y, z = xyz(i)
        ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
        return (at(x, y, z) * n + at(x + dx, y + dy, z + dz))[ok]

    i = torch.arange(n, device=_device())
    hops = [(a, b, c) for a in range(-2, 3) for b in range(-2, 3) for c in range(-2, 3) if abs(a) + abs(b) + abs(c) <= 2]
    key = torch.sort(torch.cat([pairs(i, *o) for o in hops if sum(map(abs, o)) <= 1])).values
    row, col = _parts(key, n)
    A = Mat(n, n, key, torch.where(row == col, torch.full_like(row, 6, dtype=torch.float64), d.mesh_values(key.numel())))
    if case["family"] == "static":
        return F64, A, None, [], None
    window = case["family"] == "window"
    far = [o for o in hops if sum(map(abs, o)) == 2] if window else hops
    o = torch.tensor(far, device=_device(), dtype=torch.int64)
    batches = []
    for _ in range(PAIRS):
        got, have = [], 0
        while have < case["updates"]:
            count = 2 * (case["updates"] - have) + 64
            w = o[shape.below(count, len(far))]
            got.append(pairs(shape.below(count, n), w[:, 0], w[:, 1], w[:, 2]))
            have += got[-1].numel()
        key = torch.cat(got)[:case["updates"]]
        if window:
            key = torch.unique(key)
            key = key[d.order(key.numel())]
            batches.append(_updates(key, d.mesh_values(key.numel()), torch.full_like(key, INS).to(torch.uint8), n))
        else:
            batches.append(_mixed(shape, d, key, d.mesh_values(key.numel()), n))
    return F64, A, None, _ring(A, batches), None


def _graph(case, shape, d):
    """A symmetrised R-MAT graph without self-loops, a weight per edge; batches half insertions of edges held out of it,
    half deletions of its edges, both directions of each.  For paths also the sparse B, 1 % full."""
    paths = case["family"] == "paths"
    sr = I32 if paths else case["semiring"]
    a, b, c, _ = GRAPH500 if paths else FLAT
    scale, edges = case["scale"], case.get("edges", 0)
    n, m = 1 << scale, (16 if paths else 8) << scale
    mask = int(d.below(1, n))
    u = torch.zeros(m, dtype=torch.int64, device=_device())
    v = torch.zeros_like(u)
    for level in range(scale):
        r = torch.rand(m, generator=shape.g, device=_device())
        u |= (r >= a + b).to(torch.int64) << level
        v |= (((r >= a) & (r < a + b)) | (r >= a + b + c)).to(torch.int64) << level
    keep = u != v
    e = torch.unique(torch.minimum(u, v)[keep] * n + torch.maximum(u, v)[keep])
    u, v = _parts(e, n)
    u, v, w = u ^ mask, v ^ mask, d.values(e.numel(), sr)
    pick = shape.order(e.numel())
    held = min(4 * edges, e.numel() // 20)
    out, stay = pick[:held], pick[held:]
    key, order = torch.sort(torch.cat([u[stay] * n + v[stay], v[stay] * n + u[stay]]))
    A = Mat(n, n, key, torch.cat([w[stay], w[stay]])[order])
    B = None
    if paths:
        raw = torch.unique(shape.below(int(n * case["cols"] * 0.01), n * case["cols"]))
        i, j = _parts(raw, case["cols"])
        B = Mat(n, case["cols"], torch.sort((i ^ mask) * case["cols"] + j).values, d.values(raw.numel(), sr))
    batches = []
    for _ in range(PAIRS if edges else 0):
        ni = edges // 2
        x = torch.cat([out[shape.below(ni, held)], stay[shape.below(edges - ni, stay.numel())]])
        op = torch.cat([torch.full((ni,), INS, dtype=torch.uint8, device=x.device),
                        torch.full((edges - ni,), DEL, dtype=torch.uint8, device=x.device)])
        o = shape.order(edges)
        x, op = x[o], op[o]
        two = torch.stack([u[x] * n + v[x], v[x] * n + u[x]], 1).reshape(-1)
        op = op.repeat_interleave(2)
        val = w[x].repeat_interleave(2)
        batches.append(_updates(two, torch.where(op == DEL, torch.zeros_like(val[:1]), val), op, n))
    return sr, A, B, _ring(A, batches), None


def _inputs(case, seed, shape=None):
    """The semiring, A and B (None: A again) and the rings of batches of A (and of B), as device tensors."""
    make = {"er": _scattered, "stencil": _mesh, "window": _mesh, "static": _mesh}.get(case["family"], _graph)
    return make(case, shape or _shape_of(case), _Draw(seed))


def _instances(case, seed):
    """The uneven instances of a group: scales over the range, the semirings in turn, batch sizes of every magnitude."""
    got = []
    for t in range(case["members"]):
        rng = random.Random(1000003 * case["updates"] + t)
        sub = {"family": "square", "scale": rng.randint(case["lo"], case["hi"]), "semiring": F64 if t % 2 == 0 else I32,
               "edges": _log(rng, 10, case["updates"]), "member": t}
        got.append((sub, 1000003 * seed + t))
    return got


def _initial_weights(seed):
    rng = np.random.default_rng(seed)
    parts = []
    for out, fan in ((64, 4), (64, 64), (1, 64)):
        parts += [rng.uniform(-1, 1, out * fan) * math.sqrt(6.0 / fan), np.zeros(out)]
    return np.concatenate(parts).astype(np.float32)


def _size_samples(case, seed):
    """The estimator's inputs and targets for every row of a graph's square: log2(1 + .) of the length of A_i, of the
    sum, maximum and mean of the lengths of the rows it meets, and of the size of row i."""
    sr, A, _, _, _ = _inputs({"family": "build", "scale": case["scale"], "semiring": F64}, seed, _Draw(seed + 1))
    length = (A.rowptr[1:] - A.rowptr[:-1]).double()
    met = length[A.col.long()]
    total = torch.zeros_like(length).index_add_(0, A.rows, met)
    most = torch.zeros_like(length).scatter_reduce_(0, A.rows, met, "amax")
    X = torch.log2(1.0 + torch.stack([length, total, most, total / length.clamp(min=1.0)], 1)).float().contiguous()
    rp = _rows_of_product(A, A, torch.arange(A.nrows, device=A.key.device), sr)[0]
    return X, torch.log2(1.0 + (rp[1:] - rp[:-1]).double()).float()


def _pinned(count, dtype):
    return torch.empty(count, dtype=dtype, pin_memory=torch.cuda.is_available()).numpy()


def _result_arrays(handle):
    """Page-locked arrays with room to spare for the rows that the last batch changed."""
    rows, _, col, val = handle.read_affected()
    n, e = int(1.5 * rows.shape[0]) + 64, int(1.5 * col.shape[0]) + 1024
    return (_pinned(n, torch.int32), _pinned(n + 1, torch.int64), _pinned(e, torch.int32),
            _pinned(e, torch.float64 if val.dtype == np.float64 else torch.int32))


_TRAINED = {}


def _estimator(seed):
    """An estimator trained on a small graph, as a program with learned sizing keeps one."""
    if "weights" not in _TRAINED:
        _, A, _, _, _ = _inputs({"family": "build", "scale": 13, "semiring": F64}, 1)
        h = dspg.DynamicSpGEMM(A)
        X, y = h.row_features()
        est = dspg.Estimator(_initial_weights(1))
        est.train(X, y, batch=4096, steps=300, lr=5e-4)
        _TRAINED["weights"] = est.params()
        est.close()
        h.close()
    return dspg.Estimator(_TRAINED["weights"])


# ------------------------------------------------------------- the passes


def prepare(case, seed):
    f = case["family"]
    if f == "group":
        rings, handles = [], []
        for sub, s in _instances(case, seed):
            _, A, _, ring, _ = _inputs(sub, s)
            h = dspg.DynamicSpGEMM(A)
            h.reserve(max(b.row.shape[0] for b in ring))
            handles.append(h)
            rings.append(ring)
        group = dspg.Group(handles)
        st = {"handles": handles, "group": group, "rings": rings, "at": 0}
        for k in range(WARM):
            group.apply([r[k % len(r)] for r in rings])
            if k == 0:
                st["out"] = [_result_arrays(h) for h in handles]
        return st
    if f == "estimator":
        X, y = _size_samples(case, seed)
        return {"est": dspg.Estimator(_initial_weights(seed)), "X": X, "y": y, "case": dict(case)}
    sr, A, B, ring, ring_b = _inputs(case, seed)
    if f == "build":
        return {"A": A}
    h = dspg.DynamicSpGEMM(A, B, bloom=bool(case.get("bloom", False)))
    if f == "static":
        return {"handle": h}
    if case.get("sizing", "bound") != "bound":
        learned = case["sizing"] == "learned"
        h.set_sizing(dspg.SIZE_LEARNED if learned else dspg.SIZE_EXACT, _estimator(seed) if learned else None)
    if not case.get("device", f != "er"):
        ring = [_on_host(b) for b in ring]
        ring_b = None if ring_b is None else [_on_host(b) for b in ring_b]
    st = {"handle": h, "ring": ring, "ring_b": ring_b, "at": 0, "family": f}
    for k in range(WARM):
        _apply(st)
        if k == 0 and f != "er":
            st["out"] = _result_arrays(h)
    st["at"] = 0
    return st


def _next(st):
    k = st["at"]
    st["at"] = k + 1
    return k


def _apply(st):
    k = _next(st)
    b = st["ring"][k % len(st["ring"])]
    b2 = None if st["ring_b"] is None else st["ring_b"][k % len(st["ring_b"])]
    if st["family"] == "window" and k % 2 == 0:
        st["handle"].apply_batch(b, algebraic=True)
    else:
        st["handle"].apply_batch(b, b2)


def run(st):
    if "est" in st:
        c, est = st["case"], st["est"]
        if c["op"] == "train":
            loss = est.train(st["X"], st["y"], batch=c["batch"], steps=c["steps"], lr=5e-4)
            return loss, est.params()
        if c["op"] == "grad":
            return est.grad(st["X"], st["y"])
        return est.predict(st["X"])
    if "group" in st:
        k = _next(st)
        st["group"].apply([r[k % len(r)] for r in st["rings"]])
        return [h.read_affected(out=o) for h, o in zip(st["handles"], st["out"])]
    if "A" in st:
        h = dspg.DynamicSpGEMM(st["A"])
        c = h.read_C_device()
        h.close()
        return c
    if "ring" not in st:
        st["handle"].recompute_all()
        return st["handle"].read_C_device()
    if st["family"] == "er":
        _apply(st)
        c = st["handle"].read_C()
        return c.rowptr, c.col, c.val
    if st["family"] == "window":
        _apply(st)
        arrived = tuple(x.copy() for x in st["handle"].read_affected(out=st["out"]))
        _apply(st)
        return arrived, st["handle"].read_affected(out=st["out"])
    k = _next(st)
    return st["handle"].apply_read_affected(st["ring"][k % len(st["ring"])], out=st["out"])[1]


# ------------------------------------------------ the same in 64 bits, plainly


def _after(A, b):
    """A with b applied (the last write of a key counts), and the keys that it really changed."""
    key, order = torch.sort(b.key, stable=True)
    last = torch.ones_like(key, dtype=torch.bool)
    last[:-1] = key[1:] != key[:-1]
    key, order = key[last], order[last]
    op, val = b.op[order], b.val[order]
    at = torch.searchsorted(A.key, key).clamp(max=A.key.numel() - 1)
    there = A.key[at] == key
    gone = torch.zeros_like(A.key, dtype=torch.bool)
    gone[at[there]] = True
    write = op != DEL
    k2, o2 = torch.sort(torch.cat([A.key[~gone], key[write]]))
    return Mat(A.nrows, A.ncols, k2, torch.cat([A.val[~gone], val[write]])[o2]), key[write | there]


def _changed_rows(A, B2, b_is_a, star_a, star_b, entries):
    """Rows of C that the changes can reach; with `entries` only those that some product of a change reaches."""
    hit = torch.zeros(A.nrows, dtype=torch.bool, device=A.key.device)
    i, k = _parts(star_a, A.ncols)
    if entries:
        i = i[(B2.rowptr[k + 1] - B2.rowptr[k]) > 0]
    hit[i] = True
    star = star_a if b_is_a else star_b
    if star is not None:
        touched = torch.zeros(B2.nrows, dtype=torch.bool, device=A.key.device)
        touched[_parts(star, B2.ncols)[0]] = True
        hit[A.rows[touched[A.col.long()]]] = True
    return torch.nonzero(hit).reshape(-1)


def _rows_of_product(A, B, rows, sr):
    """(rowptr, col, val) of the given rows of A B."""
    dev = A.key.device
    number = torch.full((A.nrows,), -1, dtype=torch.int64, device=dev)
    number[rows] = torch.arange(rows.numel(), device=dev)
    sel = torch.nonzero(number[A.rows] >= 0).reshape(-1)
    k = A.col[sel].long()
    lens = B.rowptr[k + 1] - B.rowptr[k]
    src = torch.arange(sel.numel(), device=dev).repeat_interleave(lens)
    start = torch.cumsum(lens, 0) - lens
    q = B.rowptr[k][src] + torch.arange(src.numel(), device=dev) - start[src]
    key = number[A.rows[sel]][src] * B.ncols + B.col[q].long()
    prod = A.val[sel][src] * B.val[q] if sr == F64 else A.val[sel][src] + B.val[q]
    out, place = torch.unique(key, return_inverse=True)
    if sr == F64:
        val = torch.zeros(out.numel(), dtype=torch.float64, device=dev).index_add_(0, place, prod)
    else:
        val = torch.full((out.numel(),), 2 ** 31 - 1, dtype=torch.int32, device=dev)
        val.scatter_reduce_(0, place, prod, "amin")
    r, col = _parts(out, B.ncols)
    rp = torch.zeros(rows.numel() + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=rows.numel()), 0)
    return rp, col.to(torch.int32), val


def _exact_affected(sr, A, B, b, b2, entries):
    A2, star_a = _after(A, b)
    B2, star_b = (A2, None) if B is None else (B, None) if b2 is None else _after(B, b2)
    rows = _changed_rows(A, B2, B is None, star_a, star_b, entries)
    return (rows.to(torch.int32),) + _rows_of_product(A2, B2, rows, sr), A2


def _exact_estimator(case, seed):
    X, y = (x.double() for x in _size_samples(case, seed))
    dev = X.device
    w = torch.tensor(_initial_weights(seed).astype(np.float64), device=dev)  # a step keeps them in 32 bits
    cut = [0, 256, 320, 4416, 4480, 4544, 4545]

    def forward(w, X, grad):
        r = w.float().bfloat16().double().requires_grad_(grad)
        W1, b1, W2, b2, W3, b3 = (r[a:b] for a, b in zip(cut[:-1], cut[1:]))
        h1 = torch.relu(X @ W1.reshape(64, 4).T + b1)
        h2 = torch.relu(h1 @ W2.reshape(64, 64).T + b2)
        return h2 @ W3 + b3, r

    if case["op"] == "predict":
        return forward(w, X, False)[0]
    if case["op"] == "grad":
        o, r = forward(w, X, True)
        loss = ((o - y) ** 2).mean()
        loss.backward()
        return float(loss.detach()), r.grad
    n, batch = X.shape[0], case["batch"]
    nb = -(-n // batch)
    for s in range(case["steps"]):
        lo = (s % nb) * batch
        o, r = forward(w, X[lo:lo + batch], True)
        ((o - y[lo:lo + batch]) ** 2).mean().backward()
        w = (w - 5e-4 * r.grad).float().double()
    return None, w


def exact(case, seed):
    f = case["family"]
    if f == "estimator":
        return _exact_estimator(case, seed)
    if f == "group":
        got = []
        for sub, s in _instances(case, seed):
            sr, A, B, ring, _ = _inputs(sub, s)
            got.append(_exact_affected(sr, A, B, ring[0], None, False)[0])
        return got
    sr, A, B, ring, ring_b = _inputs(case, seed)
    if f in ("static", "build"):
        return _rows_of_product(A, A, torch.arange(A.nrows, device=A.key.device), sr)
    b2 = None if ring_b is None else ring_b[0]
    if f == "er":
        A2 = _after(A, ring[0])[0]
        B2 = A2 if B is None else _after(B, b2)[0]
        return _rows_of_product(A2, B2, torch.arange(A.nrows, device=A.key.device), sr)
    first, A2 = _exact_affected(sr, A, B, ring[0], b2, bool(case.get("bloom")) or f == "window")
    if f == "window":
        return first, _exact_affected(sr, A2, None, ring[1], None, False)[0]
    return first


# ----------------------------------------------------- what a pass needs


def _product_work(sr, A, B, rows, batch, mesh):
    """Bytes and operations of bringing `rows` of A B up to date and handing them out: the rows of A and the rows of B
    they use read once, C's rows written once in the handle and once to the caller."""
    s = 12 if sr == F64 else 8
    sel = torch.zeros(A.nrows, dtype=torch.bool, device=A.key.device)
    sel[rows] = True
    k = A.col[sel[A.rows]].long()
    lens = B.rowptr[k + 1] - B.rowptr[k]
    products = int(lens.sum())
    used = torch.unique(k)
    b_entries = int((B.rowptr[used + 1] - B.rowptr[used]).sum())
    number = torch.cumsum(sel, 0) - 1
    per = torch.zeros(max(rows.numel(), 1), dtype=torch.float64, device=A.key.device)
    per.index_add_(0, number[A.rows[sel[A.rows]]], lens.double())
    m = float(B.ncols)
    # the 49 products of a row of the mesh operator's square fall on 25 columns; elsewhere, columns drawn uniformly
    entries = 25.0 / 49.0 * products if mesh else float((m * -torch.expm1(-per / m)).sum())
    return {"bytes": batch * (s + 5) + s * (k.numel() + b_entries) + 36.0 * rows.numel() + 2.0 * s * entries,
            "flops": 2.0 * products}


def work(case):
    f = case["family"]
    if f == "estimator":
        per_row = 2 * (4 * 64 + 64 * 64 + 64)
        n = 1 << case["scale"]
        if case["op"] == "train":
            seen = case["steps"] * min(case["batch"], n)
            return {"bytes": 20.0 * (seen + n) + 4545 * 10.0 * case["steps"], "flops": per_row * (3.0 * seen + n)}
        return {"bytes": 20.0 * n, "flops": per_row * n * (3.0 if case["op"] == "grad" else 1.0)}
    if f == "group":
        parts = [work(sub) for sub, _ in _instances(case, 1)]
        return {x: sum(p[x] for p in parts) for x in ("bytes", "flops")}
    mesh = f in ("stencil", "static", "window")
    sr, A, B, ring, ring_b = _inputs(case, 1)
    every = torch.arange(A.nrows, device=A.key.device)
    if f in ("static", "build"):
        return _product_work(sr, A, A, every, 0, mesh)
    b2 = None if ring_b is None else ring_b[0]
    A2, star_a = _after(A, ring[0])
    B2, star_b = (A2, None) if B is None else (B, None) if b2 is None else _after(B, b2)
    rows = _changed_rows(A, B2, B is None, star_a, star_b, False)
    count = ring[0].row.shape[0] + (0 if b2 is None else b2.row.shape[0])
    got = _product_work(sr, A2, B2, rows, count, mesh)
    if f == "er":  # the whole of C is handed out
        whole = _product_work(sr, A2, B2, every, 0, mesh)
        got["bytes"] += whole["bytes"] / 2
    if f == "window":  # a batch and its expiry
        got = {x: 2 * got[x] for x in got}
    return got


def tolerance(case):
    f = case["family"]
    if f == "estimator":
        # 32-bit sums over rows in another order, and a weight that rounds to the other bfloat16 neighbour in training
        return {"rel": 4e-6, "max": 4e-4} if case["op"] == "predict" else {"rel": 2e-5, "max": 2e-3}
    # (min,+) on whole numbers is exact; (+,.) in 64 bits in any order: two runs differ by 1.3e-16 and either is up to
    # 2.8e-16 from the exact values, single entries by 8e-16; entries whose terms cancel may differ by more
    sr = case.get("semiring", I32 if f == "paths" else F64)
    return "exact" if sr == I32 and f != "group" else {"rel": 2e-15, "max": 2e-14}
