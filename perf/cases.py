"""The builds that programs using this library ask for, as timed cases.

A case says which entry point is called (``op``) and on what: point counts,
point distributions, tree depth ``level`` or cluster size ``s``, and options.

A case's geometry is its own; the seed chooses one of the 48 symmetries of
the cube and the order of the points.  So every seed gives other inputs and
other trees of the same sizes.

Outputs are whole trees.  Deep trees have more arrays than are handy to pass
around one by one: some kinds then come as one array, all levels one after
another.  Batched and served builds are used through the C structs' device
pointers (``raw=True``, or the server's own trees), so their arrays are
gathered only when somebody reads them (:class:`Gathered`).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1301_1704_gb300 import fmmds

KINDS = ("uniform", "sphere", "clumps", "wide", "mixed")


def listed():
    return [
        # A small problem: every launch and host step counts.
        {"name": "small", "op": "build", "n": 16384, "m": 16384, "src": "uniform",
         "recv": "uniform", "level": 4},
        # A handful of small clusters of uneven size in one call, each to its own depth.
        {"name": "small_batch", "op": "batch", "sets": 24, "lo": 50, "hi": 40000, "s": 64},
        # An ordinary evaluation grid: odd sizes, sources and receivers shaped differently.
        {"name": "ragged", "op": "build", "n": 300001, "m": 200003, "src": "uniform",
         "recv": "wide", "level": 6},
        # A time step of an N-body system: the same clustered points as sources and
        # receivers, rebuilt from the same buffers in graph mode.
        {"name": "time_step", "op": "self", "n": 1000000, "src": "clumps", "level": 9,
         "graphs": True},
        # A boundary-element surface against a clustered cloud, depth left to the cluster size.
        {"name": "cluster_size", "op": "build", "n": 1000000, "m": 700001, "src": "sphere",
         "recv": "clumps", "s": 64},
        # The large uniform problem, sources and receivers drawn apart.
        {"name": "uniform", "op": "build", "n": 1 << 24, "m": 1 << 24, "src": "uniform",
         "recv": "uniform", "level": 7},
        # The large sparse octree: most boxes empty, a few very full.
        {"name": "sparse", "op": "build", "n": 1 << 24, "m": 1 << 24, "src": "mixed",
         "recv": "mixed", "level": 9},
        # Many independent problems of uneven size in one call.
        {"name": "batch", "op": "batch", "sets": 512, "lo": 1000, "hi": 1000000, "s": 64},
        # Points that arrive in pinned host memory.
        {"name": "host_input", "op": "host", "n": 1 << 24, "m": 1 << 24, "src": "uniform",
         "recv": "uniform", "level": 7},
        # The direct-sum side: sorted points, and every receiver box's near sources.
        {"name": "near_field", "op": "near", "n": 1 << 20, "m": 1 << 20, "src": "uniform",
         "recv": "uniform", "level": 6},
        # A node's view of a partitioned problem: the tree of its sources and their box types.
        {"name": "partition", "op": "types", "n": 1 << 20, "src": "wide", "level": 7, "lpar": 3,
         "nodes": 4},
        # Resident systems stepped by the server, four steps each.
        {"name": "served", "op": "serve", "sizes": "10000 10000 100000 100000 1000000 1000000",
         "levels": "7 7 8 8 9 9", "steps": 4},
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]; mostly odd ones, some powers of two."""
    if rng.random() < 0.2:
        return 1 << rng.randint(math.ceil(math.log2(lo)), int(math.log2(hi)))
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _level(rng, n, kind):
    """A fixed depth for n points: a few points a finest box where the points are."""
    base = math.log(max(n, 8) / rng.uniform(2.0, 30.0)) / math.log(8.0)
    extra = {"uniform": 0.0, "wide": 0.7, "sphere": 1.0, "mixed": 1.2, "clumps": 1.7}[kind]
    return min(9, max(2, int(round(base + extra))))


def draw(rng):
    op = rng.choices(("build", "self", "batch", "host", "near", "types", "serve"),
                     (40, 18, 16, 8, 8, 6, 4))[0]
    if op == "batch":
        hi = _size(rng, 2000, 1000000)
        most = max(4, min(512, int(40e6 / hi)))
        return {"op": op, "sets": int(round(math.exp(rng.uniform(math.log(4), math.log(most))))),
                "lo": max(20, hi // rng.choice((2, 30, 1000))), "hi": hi,
                "s": rng.choice((8, 32, 64, 64, 64, 300))}
    if op == "serve":
        k = rng.randint(2, 6)
        sizes = [_size(rng, 5000, 1000000) for _ in range(k)]
        return {"op": op, "sizes": " ".join(map(str, sizes)), "steps": rng.randint(1, 4),
                "levels": " ".join(str(min(9, _level(rng, n, "clumps") + 1)) for n in sizes)}
    src = rng.choice(KINDS)
    if op == "types":
        n = _size(rng, 5000, 1 << 21)
        level = max(3, _level(rng, n, src))
        return {"op": op, "n": n, "src": src, "level": level, "lpar": rng.randint(2, min(4, level)),
                "nodes": rng.randint(2, 8)}
    if op == "near":
        n, m = _size(rng, 2000, 1 << 20), _size(rng, 2000, 1 << 20)
        return {"op": op, "n": n, "m": m, "src": "uniform", "recv": rng.choice(("uniform", "wide")),
                "level": _level(rng, n, "uniform")}
    n = _size(rng, 1000, 1 << 24)
    case = {"op": op, "n": n, "src": src}
    if op != "self":
        case["recv"] = rng.choice((src, src, rng.choice(KINDS)))
        case["m"] = n if rng.random() < 0.4 else _size(rng, 1000, 1 << 24)
    if op == "self":
        case["graphs"] = rng.random() < 0.5
    # the depth is left to the cluster size only where a finest box can hold s points
    if op != "host" and rng.random() < 0.3 and n <= 4000000 and case.get("m", 0) <= 4000000:
        case["s"] = rng.choice((16, 64, 64, 300))
    else:
        case["level"] = _level(rng, n, src)
        if rng.random() < 0.12:
            case["order"] = "box"
    return case


# ---------------------------------------------------------------------------
# Points.

def _draw_points(gen, n, kind):
    dev = "cuda"
    if kind == "uniform":
        return torch.rand((n, 3), generator=gen, device=dev)
    if kind == "sphere":  # radius 0.4, radial jitter 1e-3
        d = torch.randn((n, 3), generator=gen, device=dev)
        r = 0.4 + 1e-3 * torch.randn((n, 1), generator=gen, device=dev)
        return 0.5 + r * d / d.norm(dim=1, keepdim=True)
    if kind == "mixed":  # half on the sphere, half in clumps
        h = n // 2
        return torch.cat([_draw_points(gen, h, "sphere"), _draw_points(gen, n - h, "clumps")])
    k, sigma = (64, 0.01) if kind == "clumps" else (8, 0.06)
    c = 0.1 + 0.8 * torch.rand((k, 3), generator=gen, device=dev)
    x = c[torch.randint(k, (n,), generator=gen, device=dev)]
    x = (x + sigma * torch.randn((n, 3), generator=gen, device=dev)).abs_()
    return torch.where(x > 1.0, 2.0 - x, x)  # folded back at the walls


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _symmetry(gen):
    """Axis order and reflected axes of one of the cube's symmetries."""
    return (torch.randperm(3, generator=gen, device="cuda"),
            torch.randint(2, (3,), generator=gen, device="cuda").bool())


def _points(gen, sym, n, kind, which=0):
    """float32 [n, 3] on the GPU, in (0, 1); `which` tells point sets of one case apart."""
    x = _draw_points(_generator(1000003 * which + 17 * n + KINDS.index(kind)), n, kind)
    # odd multiples of 2^-24: exact under x -> 1 - x, and never on a cell's border
    x = ((x * 2.0 ** 23).floor().clamp(0, 2 ** 23 - 1) * 2 + 1) * 2.0 ** -24
    axes, mirrored = sym
    x = x[torch.randperm(n, generator=gen, device="cuda")][:, axes]
    return torch.where(mirrored, 1.0 - x, x).contiguous()


def _batch_sets(case):
    """Sizes and kinds of a batch: the case's own, whatever the seed."""
    rng = np.random.default_rng(7)
    n = np.rint(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["sets"])))
    kinds = rng.integers(0, 3, case["sets"])
    return [(int(v), ("uniform", "sphere", "clumps")[k]) for v, k in zip(n, kinds)]


def prepare(case, seed):
    gen = _generator(seed)
    sym = _symmetry(gen)
    st = {"case": case}
    op = case["op"]
    if op == "serve":
        srv = fmmds.Server(0, workers=2, max_batch=8)
        st["sizes"] = [int(v) for v in case["sizes"].split()]
        st["systems"] = [srv.add_system(_points(gen, sym, n, "clumps", k), int(L), 0.1,
                                        seed=seed * 100 + k)
                         for k, (n, L) in enumerate(zip(st["sizes"], case["levels"].split()))]
        st["server"] = srv
        return st
    ctx = st["ctx"] = fmmds.Context(0)
    if op == "batch":
        pts = [_points(gen, sym, n, kind, k) for k, (n, kind) in enumerate(_batch_sets(case))]
        st["batch"] = ctx.batch([(p, p) for p in pts])
        return st
    st["src"] = _points(gen, sym, case["n"], case["src"])
    st["recv"] = _points(gen, sym, case["m"], case["recv"], 1) if "m" in case else st["src"]
    if op == "host":
        for k in ("src", "recv"):
            st[k] = st[k].cpu().pin_memory()
    if case.get("graphs"):
        ctx.set_graphs(True)
    if op == "types":
        # the boxes of the partition level dealt out in Morton order
        boxes = ctx.build(st["src"], st["src"], L=case["lpar"]).src.nbox[case["lpar"]]
        at = torch.arange(boxes, device="cuda", dtype=torch.int64)
        st["owner"] = (at * case["nodes"] // max(boxes, 1)).to(torch.int32)
    st["depth"] = {"s": case["s"]} if "s" in case else {"L": case["level"]}
    flags = {"host": fmmds.FMM_FLAG_HOST_INPUT, "near": fmmds.FMM_FLAG_SORTED_XYZ}.get(op, 0)
    st["flags"] = flags | (fmmds.FMM_FLAG_BOX_ORDER if case.get("order") == "box" else 0)
    return st


# ---------------------------------------------------------------------------
# One pass.

LISTS = ("e2_off", "e2_idx", "e4_off", "e4_idx")
BOXES = ("key", "off", "parent", "child")


def _arrays(tree, own, most):
    """A tree's arrays: both sides' (`own`: one side's, sources = receivers)
    permutation and boxes, and the lists of every level; at most `most`."""
    sides = ("src",) if own else ("src", "recv")
    L = tree.L
    count = len(sides) * (4 * L + 3) + 4 * (L - 1)
    out = {k: [getattr(tree, k)[l] for l in range(2, L + 1)] for k in LISTS}
    for name in sides:
        side = getattr(tree, name)
        out[name] = {"perm": side.perm, "key": side.key, "off": side.off,
                     "parent": side.parent[1:], "child": side.child[:-1]}
    for k in ("parent", "child", "off", "key"):
        if count > most:
            for name in sides:
                count -= len(out[name][k]) - 1
                out[name][k] = torch.cat(out[name][k])
    return out


class Arrays(dict):
    """Arrays that live in a context's memory, and what keeps that context."""

    def __init__(self, arrays, owner):
        super().__init__(arrays)
        self.owner = owner


class Gathered(Arrays):
    """The arrays of several trees, each kind in one tensor, gathered when
    read.  `room`: entries a point that a kind's tensor has room for, where the
    trees' sizes follow from the time step (the rest is zero)."""

    KEYS = ("perm",) + BOXES + LISTS

    def __init__(self, owner, trees, points=0, room=None):
        super().__init__(dict.fromkeys(self.KEYS), owner)
        self._trees, self._points, self._room = trees, points, room

    def __getitem__(self, kind):
        parts = []
        for tree in self._trees():
            a = _arrays(tree, True, 1 << 30)
            v = a[kind] if kind in LISTS else a["src"][kind]
            # copied: a served tree's arrays may move when the next one is asked for
            parts.append(torch.cat(v) if isinstance(v, list) else v.clone())
        x = torch.cat(parts)
        if self._room:
            y = torch.zeros(self._points * self._room[kind] + 1024, dtype=x.dtype, device=x.device)
            y[:x.numel()] = x
            return y
        return x

    def items(self):
        return [(k, self[k]) for k in self.KEYS]

    def values(self):
        return [self[k] for k in self.KEYS]


ROOM = {"perm": 1, "key": 10, "off": 10, "parent": 10, "child": 10,
        "e2_off": 10, "e2_idx": 80, "e4_off": 10, "e4_idx": 400}


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "serve":
        srv, systems = state["server"], state["systems"]
        ids = [srv.submit(k) for _ in range(case["steps"]) for k in systems]
        infos = [srv.wait(i) for i in ids]
        return {"entries": [i["nnz_e4"] for i in infos[-len(systems):]],
                "trees": Gathered(state, lambda: (srv.tree(k) for k in systems),
                                  sum(state["sizes"]), ROOM)}
    ctx = state["ctx"]
    if op == "batch":
        b = state["batch"]
        outs = ctx.build_batched(b, s=case["s"], raw=True)
        return Gathered(state, lambda: (fmmds._tree_from(outs[i], *b.sizes[i]) for i in range(b.k)))
    tree = ctx.build(state["src"], state["recv"], flags=state["flags"], **state["depth"])
    extra = {}
    if op == "near":
        off, pts = ctx.gather_e2(tree, tree.L)
        extra = {"sorted_src": tree.sorted_src, "sorted_recv": tree.sorted_recv,
                 "near_off": off, "near": pts}
    if op == "types":
        extra = {"types": ctx.box_types(tree, case["lpar"], state["owner"], 1)}
    own = state["recv"] is state["src"]
    most = 64 - (4 if op == "near" else tree.L if op == "types" else 0)
    return Arrays({**_arrays(tree, own, most), **extra}, state)


# ---------------------------------------------------------------------------
# What a pass cannot do without: its points read once, its arrays written
# once.  How many boxes and list entries there are follows from the points,
# so one build counts them.

def _bytes(v):
    if isinstance(v, torch.Tensor):
        return v.numel() * v.element_size()
    if isinstance(v, dict):
        return sum(_bytes(x) for x in v.values())
    return sum(_bytes(x) for x in v) if isinstance(v, (list, tuple)) else 0


def work(case):
    state = prepare(case, 1)
    out = run(state)
    if case["op"] == "serve":  # every step moves the points and writes the tree anew
        points = sum(state["sizes"])
        total = sum(_bytes(_arrays(state["server"].tree(k), True, 1 << 30)) for k in state["systems"])
        return {"bytes": case["steps"] * (total + 24 * points), "flops": 0}
    total = _bytes(out)
    if case["op"] == "batch":
        points = sum(n for n, _ in _batch_sets(case))
    else:
        points = case["n"] + case.get("m", 0)
    return {"bytes": total + 12 * points, "flops": 0}


# ---------------------------------------------------------------------------
# All outputs but the sorted and gathered points are whole numbers.

def _keys(x):
    """63-bit Morton keys of float64 points."""
    q = (x * 2.0 ** 21).floor().clamp(0, 2 ** 21 - 1).to(torch.int64)
    key = torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return key


def _sorted(x):
    key = _keys(x)
    order = torch.argsort(key, stable=True)
    return x[order], key[order]


def exact(case, seed):
    if case["op"] != "near":
        return None
    gen = _generator(seed)
    sym = _symmetry(gen)
    src = _points(gen, sym, case["n"], case["src"]).double()
    recv = _points(gen, sym, case["m"], case["recv"], 1).double()
    L = case["level"]
    src, skey = _sorted(src)
    recv, rkey = _sorted(recv)
    skey, rkey = skey >> (63 - 3 * L), rkey >> (63 - 3 * L)
    boxes = torch.unique_consecutive(rkey)
    cell = torch.stack([sum(((boxes >> (3 * b + a)) & 1) << b for b in range(L)) for a in range(3)], 1)
    # per receiver box the keys of its 27 cells in ascending order, and their points' ranges
    near = []
    for d in range(27):
        c = cell + torch.tensor([d % 3 - 1, d // 3 % 3 - 1, d // 9 - 1], device="cuda")
        ok = ((c >= 0) & (c < (1 << L))).all(dim=1)
        k = sum(((c[:, a] >> b) & 1) << (3 * b + a) for b in range(L) for a in range(3))
        near.append(torch.where(ok, k, torch.full_like(k, -1)))
    near = torch.stack(near, 1).sort(dim=1).values.reshape(-1)
    first = torch.searchsorted(skey, near)
    count = torch.searchsorted(skey, near, right=True) - first
    end = count.cumsum(0)
    total = int(end[-1])
    at = torch.repeat_interleave(first - (end - count), count, output_size=total)
    pts = src[at + torch.arange(total, device="cuda")]
    return {"near": pts, "sorted_recv": recv, "sorted_src": src}
