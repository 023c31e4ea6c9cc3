"""Workloads that the speed of this library is measured on.

Each case is a dict of plain values.  `what` names the call that a program
makes, the other values its sizes:

  run       cs.run: sprinkle, relate, count and actions on device buffers
  evaluate  cs.evaluate: one set, results on the host (coords: the caller
            brings the coordinates, else the set is sprinkled from its seed)
  batch     cs.Batch.launch: a planned ensemble of Poisson-sized sets
  serve     serve.Server.run: requests that are all there, continuous batching
  layers    cs.layer_sums + cs.dalembertian with a field, on a causal matrix
  relate    cs.causal_matrix alone, from sorted coordinates
  lists     cs.degrees and both sparse relation lists (C entry points) of a causal matrix
  chains    cs.longest_chain (whole set, one pair) and cs.greedy_antichain
"""
from __future__ import annotations

import functools
import math
from decimal import Decimal, localcontext

import numpy as np
import torch

import paper_1805_04463_gb300 as cs
from paper_1805_04463_gb300 import serve

EPS = (0.0, 0.05, 0.1, 0.2)  # the local action and three smeared ones

ORDER, DIAMOND2, DIAMOND4, DIAMOND3, SLAB, SQUARE, CYLINDER = range(7)
DIMS = {ORDER: 2, DIAMOND2: 2, DIAMOND4: 4, DIAMOND3: 3, SLAB: 2, SQUARE: 2, CYLINDER: 2}


def listed():
    return [
        # the smallest whole evaluation: latency and launches count
        {"name": "run_2d_order_1024", "what": "run", "kind": ORDER, "n": 1024},
        # a 3+1 sprinkling of the usual size
        {"name": "run_4d_diamond_16384", "what": "run", "kind": DIAMOND4, "n": 16384},
        # the large set of the benchmark (2.1 GB of bitset)
        {"name": "run_2d_order_131072", "what": "run", "kind": ORDER, "n": 131072},
        # one de Sitter slab to the host, as a script that averages over seeds calls it; an odd size
        {"name": "evaluate_ds_slab_4099", "what": "evaluate", "kind": SLAB, "n": 4099, "coords": False},
        # a program's own 2+1 coordinates in, abundances and actions out
        {"name": "evaluate_3d_coords_20011", "what": "evaluate", "kind": DIAMOND3, "n": 20011, "coords": True},
        # the ensemble of the benchmark: 512 1+1 diamonds of about 4096 elements, 256 3+1 ones of about 2048
        {"name": "batch_768", "what": "batch", "kind": DIAMOND2, "sets": 512, "mean": 4096, "kind2": DIAMOND4,
         "sets2": 256, "mean2": 2048},
        # a chunk of the ensemble driver with small sets
        {"name": "batch_small_256", "what": "batch", "kind": SLAB, "sets": 160, "mean": 600, "kind2": DIAMOND3,
         "sets2": 96, "mean2": 300},
        # a burst of requests for the server, over its range of sizes
        {"name": "serve_burst_24", "what": "serve", "requests": 24, "log2_min": 10.0, "log2_max": 16.0},
        # the scalar field operator on a 3+1 set
        {"name": "layers_4d_diamond_8192", "what": "layers", "kind": DIAMOND4, "n": 8192},
        # the causal matrix of a de Sitter slab at the thesis's larger sizes, ragged
        {"name": "relate_ds_slab_50021", "what": "relate", "kind": SLAB, "n": 50021},
        # degree vectors and relation lists of a 1+1 set
        {"name": "lists_2d_diamond_30011", "what": "lists", "kind": DIAMOND2, "n": 30011},
        # height, one pair's chain and an antichain of a 2D order
        {"name": "chains_2d_order_32768", "what": "chains", "kind": ORDER, "n": 32768},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["run", "run", "evaluate", "batch", "serve", "layers", "relate", "lists", "chains"])
    kind = rng.choice(list(DIMS))
    if what == "run":
        return {"what": what, "kind": kind, "n": _log(rng, 256, 131072)}
    if what == "evaluate":
        return {"what": what, "kind": kind, "n": _log(rng, 256, 40000), "coords": rng.random() < 0.5}
    if what == "batch":
        mean = _log(rng, 200, 5000)
        return {"what": what, "kind": kind, "sets": _log(rng, 8, 512), "mean": mean, "kind2": rng.choice(list(DIMS)),
                "sets2": _log(rng, 4, 256), "mean2": max(100, int(mean * rng.uniform(0.4, 1.0)))}
    if what == "serve":
        return {"what": what, "requests": rng.randint(4, 32), "log2_min": 10.0, "log2_max": rng.uniform(12.0, 16.0)}
    if what == "layers":
        return {"what": what, "kind": kind, "n": _log(rng, 700, 30000)}
    if what == "relate":
        return {"what": what, "kind": kind, "n": _log(rng, 1000, 131072)}
    if what == "lists":
        return {"what": what, "kind": kind, "n": _log(rng, 1000, 60000)}
    return {"what": what, "kind": kind, "n": _log(rng, 1000, 40000)}


# ------------------------------------------------------------------ inputs

def _set_seed(seed, s=0):
    return (int(seed) * 1_000_003 + 7919 * s + 0xC5E70000) & 0x7FFFFFFFFFFFFFFF


def _batch_sets(case, seed):
    """The sizes follow from the case alone, the sets from the seed."""
    rng = np.random.default_rng([case["mean"], case["mean2"], case["sets"], case["sets2"]])
    sizes = list(rng.poisson(case["mean"], case["sets"])) + list(rng.poisson(case["mean2"], case["sets2"]))
    kinds = [case["kind"]] * case["sets"] + [case["kind2"]] * case["sets2"]
    return [(k, max(int(n), 1), _set_seed(seed, s)) for s, (k, n) in enumerate(zip(kinds, sizes))]


def _requests(case, seed):
    """Sizes are the middles of equal slices of the log range, in a seeded order: every seed asks
    for the same work."""
    rng = np.random.default_rng(int(seed))
    m, lo, hi = case["requests"], case["log2_min"], case["log2_max"]
    sizes = [int(2.0 ** (lo + (hi - lo) * (s + 0.5) / m)) for s in range(m)]
    return [(0.0, ORDER if s % 2 else DIAMOND4, sizes[p], _set_seed(seed, s)) for s, p in enumerate(rng.permutation(m))]


def _field(case, seed):
    return np.random.default_rng(int(seed)).standard_normal(case["n"])


def _matrix(kind, n, seed):
    """A set's causal matrix, with the buffers it came through given back."""
    coords = torch.empty((cs.dim(kind), n), dtype=torch.int32, device="cuda")
    ws = torch.empty(cs.sprinkle_workspace_bytes(kind, n), dtype=torch.uint8, device="cuda")
    cs.sprinkle(kind, n, seed, coords, ws)
    bits = torch.empty((n, cs.row_words(n)), dtype=torch.int64, device="cuda")
    cs.causal_matrix(kind, n, coords, bits)
    return coords, bits


def prepare(case, seed):
    s = dict(case)
    what = case["what"]
    if what == "batch":
        s["batch"] = cs.Batch(_batch_sets(case, seed), n_eps=len(EPS))
    elif what == "serve":
        s["server"] = serve.Server(eps=EPS)
        s["list"] = _requests(case, seed)
    elif what == "run":
        s["buf"], s["seed"] = cs.allocate(case["kind"], case["n"]), _set_seed(seed)
    elif what == "evaluate":
        s["seed"] = _set_seed(seed)
        if case["coords"]:
            xy = torch.empty((cs.dim(case["kind"]), case["n"]), dtype=torch.int32, pin_memory=True)
            xy.copy_(_matrix_coords(case["kind"], case["n"], _set_seed(seed)))
            s["coords"] = xy.numpy()
            s["pinned"] = xy
        else:
            s["coords"] = None
        s["hist"] = torch.empty(cs.hist_len(case["n"]), dtype=torch.int64, pin_memory=True).numpy()
    else:
        n = case["n"]
        coords, bits = _matrix(case["kind"], n, _set_seed(seed))
        if what == "relate":
            s["coords"] = coords
        s["bits"] = bits
        if what == "layers":
            kmax = 3 if DIMS[case["kind"]] == 4 else 2
            s["phi"] = torch.from_numpy(_field(case, seed)).cuda()
            s["hist"] = torch.empty(cs.hist_len(n), dtype=torch.int64, device="cuda")
            s["layer"] = torch.empty((kmax + 1, n), dtype=torch.float64, device="cuda")
            s["out"] = torch.empty(n, dtype=torch.float64, device="cuda")
            s["ws"] = torch.empty(cs.interval_abundance_workspace(n), dtype=torch.uint8, device="cuda")
        elif what == "lists":
            s["kin"] = torch.empty(n, dtype=torch.int32, device="cuda")
            s["kout"] = torch.empty(n, dtype=torch.int32, device="cuda")
            s["ws"] = torch.empty(cs.lib().cs_sparse_workspace_bytes(n), dtype=torch.uint8, device="cuda")
            for side in ("past", "future"):  # room for every pair: no size has to come back to the host
                s[side] = (torch.empty(n + 1, dtype=torch.int64, device="cuda"),
                           torch.zeros(n * (n - 1) // 2, dtype=torch.int32, device="cuda"))
    return s


def _matrix_coords(kind, n, seed):
    coords = torch.empty((cs.dim(kind), n), dtype=torch.int32, device="cuda")
    ws = torch.empty(cs.sprinkle_workspace_bytes(kind, n), dtype=torch.uint8, device="cuda")
    cs.sprinkle(kind, n, seed, coords, ws)
    return coords.cpu()


def _lists(n, bits, direction, offsets, cols, ws):
    """One side's relation lists through the C entry points, into buffers of the program's own."""
    L, stream = cs.lib(), torch.cuda.current_stream().cuda_stream
    rc = L.cs_sparse_offsets(n, bits.data_ptr(), bits.shape[1], direction, offsets.data_ptr(), ws.data_ptr(),
                             ws.numel(), stream)
    if rc == 0:
        rc = L.cs_sparse_columns(n, bits.data_ptr(), bits.shape[1], direction, offsets.data_ptr(), cols.data_ptr(),
                                 cols.numel(), ws.data_ptr(), ws.numel(), stream)
    if rc != 0:
        raise cs.CsError(rc, "sparse lists")


def run(s):
    what = s["what"]
    if what == "run":
        b = s["buf"]
        cs.run(b, s["seed"], eps=EPS)
        return {"coords": b.coords, "bits": b.bits, "hist": b.hist, "actions": b.actions[:len(EPS)],
                "bracket": b.bracket}
    if what == "evaluate":
        hist, actions, bracket = cs.evaluate(s["kind"], s["n"], seed=s["seed"], coords_host=s["coords"], eps=EPS,
                                             hist_out=s["hist"])
        return {"hist": hist, "actions": np.array(actions), "bracket": bracket}
    if what == "batch":
        b = s["batch"]
        b.launch(EPS)
        return {"hist": b.hist, "actions": b.actions, "brackets": b.brackets}
    if what == "serve":
        _, results = s["server"].run(s["list"], realtime=False)
        order = sorted(results)
        return {"hist": np.concatenate([results[r][0] for r in order]),
                "actions": np.stack([results[r][1] for r in order])}
    n, bits = s["n"], s["bits"]
    if what == "relate":
        cs.causal_matrix(s["kind"], n, s["coords"], bits)
        return bits
    if what == "layers":
        cs.layer_sums(n, bits, s["hist"], s["layer"], s["layer"].shape[0] - 1, phi=s["phi"], workspace=s["ws"])
        cs.dalembertian(cs.dim(s["kind"]), n, s["layer"], s["out"], phi=s["phi"])
        return {"hist": s["hist"], "layer": s["layer"], "out": s["out"]}
    if what == "lists":
        cs.degrees(n, bits, s["kin"], s["kout"])
        for direction, side in enumerate(("past", "future")):
            _lists(n, bits, direction, *s[side], s["ws"])
        return {"in": s["kin"], "out": s["kout"], "past": s["past"], "future": s["future"]}
    height = cs.longest_chain(n, bits)
    pair = cs.longest_chain(n, bits, n // 50, n - 1 - n // 50)
    size, members = cs.greedy_antichain(n, bits, n // 2)
    return {"height": height, "pair": pair, "size": size, "members": members}


# -------------------------------------------------------------- least work

#: Share of the pairs of elements that are related, for the length of the relation lists.
_RELATED = {ORDER: 0.5, DIAMOND2: 0.5, DIAMOND4: 0.1, DIAMOND3: 8 / 35, SLAB: 0.36, SQUARE: 0.5, CYLINDER: 0.212}


def _bits_bytes(n):
    return n * ((n + 1023) // 1024) * 128


def _terms(n):
    """Flops of the interval counts: one multiply-add for each i < k < j."""
    return n * (n - 1.0) * (n - 2.0) / 3.0


def work(case):
    what = case["what"]
    if what == "batch":
        sizes = [case["mean"]] * case["sets"] + [case["mean2"]] * case["sets2"]
        return {"bytes": sum(8.0 * n + 8 * len(EPS) + 8 for n in sizes), "flops": sum(map(_terms, sizes))}
    if what == "serve":
        sizes = [n for _, _, n, _ in _requests(case, 0)]
        return {"bytes": sum(8.0 * n + 8 * len(EPS) for n in sizes), "flops": sum(map(_terms, sizes))}
    n, d = case["n"], DIMS[case["kind"]]
    coords, hist, bits = 4.0 * d * n, 8.0 * n, float(_bits_bytes(n))
    if what == "run":
        return {"bytes": coords + bits + hist, "flops": _terms(n)}
    if what == "evaluate":
        return {"bytes": hist + (coords if case["coords"] else 0.0), "flops": _terms(n)}
    if what == "relate":
        return {"bytes": coords + bits, "flops": n * (n - 1.0) / 2.0 * (2 * d)}
    if what == "layers":
        return {"bytes": bits + hist + 8.0 * n * (6 if d == 4 else 5), "flops": _terms(n)}
    if what == "lists":
        return {"bytes": bits + 24.0 * n + 2 * 4.0 * _RELATED[case["kind"]] * n * (n - 1.0) / 2.0, "flops": 0.0}
    return {"bytes": bits, "flops": 0.0}


# ------------------------------------- the same results, without the library

_M64 = (1 << 64) - 1


def _mix(z):
    """SplitMix64's output function (Steele, Lea and Flood 2014) on uint64 arrays."""
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


_GAMMA = 0x9E3779B97F4A7C15


def _draws(seed, stream, e, slot):
    state = _mix(np.array([(seed + (stream + 1) * _GAMMA) & _M64], dtype=np.uint64))
    return _mix(state + (e.astype(np.uint64) * np.uint64(65536) + np.uint64(slot + 1)) * np.uint64(_GAMMA))


def _ranks(key):
    r = np.empty(len(key), dtype=np.int64)
    r[np.argsort(key, kind="stable")] = np.arange(len(key))
    return r


@functools.lru_cache(maxsize=None)
def _slab_cells():
    unit, g = 2.0 * math.pi / 1048576.0, 83443
    t0 = math.tan((g + 0.5) * unit)
    return np.array([int((math.tan((i - g + 0.5) * unit) + t0) / (2.0 * t0) * 9007199254740992.0)
                     for i in range(2 * g + 1)], dtype=np.uint64)


def _sprinkled(kind, n, seed):
    """Time-sorted integer coordinates (dim, n) of a set, by the documented generator."""
    e = np.arange(n)

    def top(stream, slot, bits, who=e):
        return (_draws(seed, stream, who, slot) >> np.uint64(64 - bits)).astype(np.int64)

    if kind == ORDER:
        ru, rv = _ranks(_draws(seed, 0, e, 0)), _ranks(_draws(seed, 1, e, 0))
        c = np.empty((2, n), dtype=np.int64)
        c[0], c[1][ru] = e, rv
        return c
    if kind == DIAMOND2:
        c = np.stack([top(2, 0, 31), top(2, 1, 31)])
        key = c[0] + c[1]
    elif kind == SQUARE:
        t, x = top(6, 0, 30) - (1 << 29), top(6, 1, 30) - (1 << 29)
        c = np.stack([t + x, t - x]) + (1 << 30)
        key = c[0] + c[1]
    elif kind == CYLINDER:
        big = 683565275  # floor(2^31 / pi)
        t = ((top(7, 1, 32).astype(np.uint64) * np.uint64(2 * big)) >> np.uint64(32)).astype(np.int64) - big
        c, key = np.stack([t, top(7, 0, 32)]), t
    elif kind == SLAB:
        cell = np.searchsorted(_slab_cells(), _draws(seed, 5, e, 1) >> np.uint64(11), side="right")
        t = (cell.astype(np.int64) - 83443) * 4096 - 2048 + top(5, 2, 12)
        c, key = np.stack([t, top(5, 0, 32)]), t
    else:
        d, stream, unit = (4, 3, 1 << 20) if kind == DIAMOND4 else (3, 4, 1 << 20)
        c, left, a = np.zeros((d, n), dtype=np.int64), e, 0
        while len(left):
            q = np.stack([top(stream, d * a + k, 20, left) for k in range(d)])
            q[1:] -= unit // 2
            ok = (q[1:] ** 2).sum(0) < np.minimum(q[0], unit - q[0]) ** 2
            c[:, left[ok]] = q[:, ok]
            left, a = left[~ok], a + 1
        key = c[0]
    return c[:, np.argsort(key, kind="stable")]


def _relation(kind, coords):
    """The strict upper triangle of the causal matrix as 0/1 floats, on the GPU."""
    x = torch.from_numpy(np.ascontiguousarray(coords)).cuda()
    n = x.shape[1]
    out = torch.empty((n, n), dtype=torch.float32, device="cuda")
    after = torch.arange(n, device="cuda")
    for i in range(0, n, 1024):
        d = x[:, None, :] - x[:, i:i + 1024, None]
        if kind in (ORDER, DIAMOND2, SQUARE):
            rel = (d[0] > 0) & (d[1] > 0)
        elif kind in (SLAB, CYLINDER):
            turn = d[1] & 0xFFFFFFFF
            rel = torch.minimum(turn, (1 << 32) - turn) < d[0].abs()
        else:
            rel = d[0] ** 2 - (d[1:] ** 2).sum(0) > 0
        out[i:i + 1024] = (rel & (after[None, :] > after[i:i + 1024, None])).float()
    return out


def _counted(c):
    """Blocks (first row, relation, interval sizes): 0/1 products summed in float32 are exact below 2^24."""
    for i in range(0, c.shape[0], 2048):
        yield i, c[i:i + 2048] > 0, c[i:i + 2048] @ c


def _abundances(c):
    n = c.shape[0]
    hist = torch.zeros(max(n - 1, 1), dtype=torch.int64, device="cuda")
    for _, rel, m in _counted(c):
        hist += torch.bincount(m[rel].long(), minlength=len(hist))
    return hist.cpu().numpy()


@functools.lru_cache(maxsize=32)
def _smearing(dim, eps, length):
    """f_d(k, eps) for k < length, as decimals; the list ends where (1 - eps)^k has become negligible."""
    with localcontext() as ctx:
        ctx.prec = 60
        e = Decimal(eps)
        q, p, out = 1 - e, Decimal(1), []
        for k in range(length):
            x, y, z = k * e / q, k * (k - 1) * (e / q) ** 2, k * (k - 1) * (k - 2) * (e / q) ** 3
            out.append(p * (1 - 2 * x + y / 2 if dim == 2 else 1 - 27 * x / 8 + 9 * y / 8 if dim == 3
                            else 1 - 9 * x + 8 * y - 4 * z / 3))
            p *= q
            if k > 8 and p * (1 + k) ** 3 < Decimal(10) ** -40:
                break
        return out


def _c3():
    return Decimal((math.pi / (3.0 * math.sqrt(2.0))) ** (2.0 / 3.0) / math.gamma(5.0 / 3.0))


def _bracket(dim, n, hist):
    h = [int(v) for v in hist[:4]] + [0] * 4
    return (n - 2 * h[0] + 4 * h[1] - 2 * h[2] if dim == 2 else 8 * n - 8 * h[0] + 27 * h[1] - 18 * h[2] if dim == 3
            else n - h[0] + 9 * h[1] - 16 * h[2] + 8 * h[3])


def _actions(dim, n, hist):
    out = []
    with localcontext() as ctx:
        ctx.prec = 60
        for eps in EPS:
            if eps <= 0.0:
                b = Decimal(_bracket(dim, n, hist))
                out.append(2 * b if dim == 2 else _c3() * b / 8 if dim == 3 else 4 / Decimal(6).sqrt() * b)
                continue
            e = Decimal(eps)
            total = sum((int(h) * f for h, f in zip(hist, _smearing(dim, eps, 8192)) if h), Decimal(0))
            out.append(2 * e * (n - 2 * e * total) if dim == 2
                       else _c3() * Decimal(eps ** (2.0 / 3.0)) * (n - e * total) if dim == 3
                       else 4 * (e / 6).sqrt() * (n - e * total))
        return np.array([float(v) for v in out])


def _whole(kind, n, seed):
    coords = _sprinkled(kind, n, seed)
    hist = _abundances(_relation(kind, coords))
    return coords, hist, _actions(DIMS[kind], n, hist), _bracket(DIMS[kind], n, hist)


#: Products of the plain matrix multiplications that are still done (some seconds).
_MOST = 1.2e14


def exact(case, seed):
    what = case["what"]
    if what in ("relate", "lists", "chains"):
        return None  # whole numbers only
    if what == "batch":
        sets = _batch_sets(case, seed)
        if sum(float(n) ** 3 for _, n, _ in sets) > _MOST:
            return None
        done = [_whole(*s) for s in sets]
        return {"hist": np.concatenate([d[1] for d in done]), "actions": np.stack([d[2] for d in done]),
                "brackets": np.array([d[3] for d in done])}
    if what == "serve":
        sets = [(k, n, sd) for _, k, n, sd in _requests(case, seed)]
        if sum(float(n) ** 3 for _, n, _ in sets) > _MOST:
            return None
        done = [_whole(*s) for s in sets]
        return {"hist": np.concatenate([d[1] for d in done]), "actions": np.stack([d[2] for d in done])}
    n, kind = case["n"], case["kind"]
    if float(n) ** 3 > _MOST:
        return None
    if what == "layers":
        c = _relation(kind, _sprinkled(kind, n, _set_seed(seed)))
        phi = _field(case, seed)
        kmax = 3 if DIMS[kind] == 4 else 2
        hist, layer = np.zeros(max(n - 1, 1), dtype=np.int64), np.zeros((kmax + 1, n))
        for i, rel, m in _counted(c):
            hist += torch.bincount(m[rel].long(), minlength=len(hist)).cpu().numpy()
            p = torch.from_numpy(phi[i:i + rel.shape[0]]).cuda()
            for k in range(kmax + 1):
                layer[k] += (p @ (rel & (m == k)).double()).cpu().numpy()
        s = layer
        out = (2.0 * (-phi + 2.0 * (s[0] - 2.0 * s[1] + s[2])) if DIMS[kind] == 2
               else float(_c3()) * (-phi + s[0] - 3.375 * s[1] + 2.25 * s[2]) if DIMS[kind] == 3
               else 4.0 / math.sqrt(6.0) * (-phi + s[0] - 9.0 * s[1] + 16.0 * s[2] - 8.0 * s[3]))
        return {"hist": hist, "layer": layer, "out": out}
    coords, hist, actions, bracket = _whole(kind, n, _set_seed(seed))
    if what == "evaluate":
        return {"hist": hist, "actions": actions, "bracket": bracket}
    return {"coords": None, "bits": None, "hist": hist, "actions": actions, "bracket": np.array([bracket])}
