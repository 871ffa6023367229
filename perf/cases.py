"""The measured cases: sparse permutation, extraction and assignment as a program uses them.

A case is a dict of plain values.  ``listed()`` holds the fixed ones, ``draw`` gives more
of the same ranges, ``prepare`` makes a case's matrices and index vectors on the GPU from
a seed, ``run`` makes one pass through the public entry points (``Context``), ``work``
says what a pass cannot do without, and ``exact`` computes the output values of the same
inputs in 64 bits with plain torch operations.

Matrices stand in for the graph classes the library serves: Erdos-Renyi ("er", uniformly
random columns), R-MAT ("rmat", power-law rows, optionally symmetrised) and the 2-D
5-point mesh ("mesh").  Index widths ("rp" row pointer, "ci" column, "ix" index vectors)
and value widths ("vt") are in bits.  A case's sizes, the number of stored entries of its
matrices and of its result among them, follow from the case alone: random entries are
drawn near the expected number and a few dropped (or added) to meet it, so results of
different seeds have the same shape.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2509_20776_gb300 import CSR, Context
from paper_2509_20776_gb300._binding import (SP_ASSIGN_PLUS, SP_ASSIGN_REPLACE, SP_ASSIGN_SELECT2ND, ExtractBatch)

DEV = "cuda"
_INT = {32: torch.int32, 64: torch.int64}
_FLT = {32: torch.float32, 64: torch.float64}
_MODE = {"replace": SP_ASSIGN_REPLACE, "second": SP_ASSIGN_SELECT2ND, "plus": SP_ASSIGN_PLUS}
_RMAT = (0.57, 0.19, 0.19, 0.05)

_ctx = None


def _context() -> Context:
    """The program's one context: it owns the workspace that all calls share."""
    global _ctx
    if _ctx is None:
        _ctx = Context()
    return _ctx


# ---- the cases -------------------------------------------------------------------------
def listed():
    i32 = {"rp": 32, "ci": 32, "ix": 32}
    i64 = {"rp": 64, "ci": 32, "ix": 32}  # int64 row pointers, int32 columns and indices
    return [
        # The smallest calls: one small matrix reordered, cut or patched on its own, where
        # launches, synchronisations and latency count (n = 4096, 8 entries per row, fp64).
        {"name": "permute-tiny", "op": "permute", "kind": "er", "n": 4096, "ncols": 4096, "d": 8, **i32, "vt": 64,
         "perm": "pair"},
        {"name": "extract-tiny", "op": "extract", "kind": "er", "n": 4096, "ncols": 4096, "d": 8, **i32, "vt": 64,
         "sel": "random", "nI": 1024, "nJ": 1024},
        {"name": "assign-tiny", "op": "assign", "kind": "er", "n": 4096, "ncols": 4096, "d": 8, **i32, "vt": 64,
         "sel": "random", "nI": 1024, "nJ": 1024, "bd": 4, "mode": "replace"},
        # An ordinary power-law graph of odd size put in degree order (the usual relabelling
        # before triangle counting or compression), 64-bit indices and values throughout.
        {"name": "permute-degree", "op": "permute", "kind": "rmat", "n": 1000003, "ncols": 1000003, "d": 8, "symm": True,
         "rp": 64, "ci": 64, "ix": 64, "vt": 64, "perm": "degree"},
        # The largest: a social network of 2^25 vertices (1.05 G entries) randomly relabelled
        # for load balance, P A P^T.
        {"name": "permute-social", "op": "permute", "kind": "rmat", "n": 1 << 25, "ncols": 1 << 25, "d": 16, "symm": True,
         **i64, "vt": 32, "perm": "sym"},
        # Half of the vertices of a large uniformly random graph, in random order (induced
        # subgraph sampling).
        {"name": "extract-urand", "op": "extract", "kind": "er", "n": 1 << 25, "ncols": 1 << 25, "d": 32, **i64, "vt": 32,
         "sel": "random", "nI": 1 << 24, "nJ": 1 << 24},
        # A contiguous off-diagonal block (domain decomposition, streaming a matrix in blocks).
        {"name": "extract-block", "op": "extract", "kind": "er", "n": 1 << 24, "ncols": 1 << 24, "d": 32, **i64, "vt": 32,
         "sel": "range", "nI": 1 << 22, "nJ": 1 << 22},
        # The subgraph of random vertices of a road-like mesh: rows of at most five entries, fp64.
        {"name": "extract-mesh", "op": "extract", "kind": "mesh", "n": 4900 * 4900, "ncols": 4900 * 4900, "d": 5, **i64,
         "vt": 64, "sel": "same", "nI": 4900 * 4900 // 8, "nJ": 4900 * 4900 // 8},
        # A block of a web graph replaced (a crawl's update written back into the matrix).
        {"name": "assign-web", "op": "assign", "kind": "rmat", "n": 1 << 25, "ncols": 1 << 25, "d": 24, "symm": False, **i64,
         "vt": 32, "sel": "random", "nI": 1 << 21, "nJ": 1 << 21, "bd": 8, "mode": "replace"},
        # Incremental update of a randomly relabelled matrix: weights of stored edges raised
        # and new edges added, in one fused call with the relabelling, odd size, fp64 sums.
        {"name": "update-plus", "op": "update", "kind": "rmat", "n": 1500001, "ncols": 1500001, "d": 12, "symm": True, **i64,
         "vt": 64, "sel": "random", "nI": 100003, "nJ": 100003, "bd": 8, "mode": "plus"},
        # Serving: many small extractions over resident matrices, planned once and run as
        # one batch (the replayed form of a server's round).
        {"name": "batch-extract", "op": "batch-extract", "kind": "rmat", "n": 1 << 20, "d": 6, "symm": True, **i64, "vt": 32,
         "nmats": 24, "nreq": 3000, "most": 65536},
        # Serving: a round of small permutations, planned and run in one call.
        {"name": "batch-permute", "op": "batch-permute", "kind": "rmat", "n": 1 << 16, "d": 6, "symm": True, **i64, "vt": 32,
         "nmats": 16, "nreq": 400},
    ]


def _log(rng, lo, hi):
    """An integer whose logarithm is spread evenly over [lo, hi]."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    op = rng.choice(["permute", "permute", "extract", "extract", "assign", "update", "batch-extract", "batch-permute"])
    rp, ci, ix = rng.choice([(32, 32, 32), (64, 32, 32), (64, 32, 32), (64, 64, 64), (64, 32, 64)])
    c = {"op": op, "rp": rp, "ci": ci, "ix": ix, "vt": rng.choice([32, 64])}
    if op.startswith("batch"):
        c |= {"kind": "rmat", "d": rng.choice([2, 4, 6, 8]), "symm": rng.random() < 0.7, "nmats": _log(rng, 2, 24),
              "nreq": _log(rng, 16, 2000 if op == "batch-extract" else 300),
              "n": _log(rng, 2000, 1 << 19 if op == "batch-extract" else 1 << 16)}
        if op == "batch-extract":
            c["most"] = _log(rng, 64, 65536)
        return c
    kind = rng.choice(["er", "er", "rmat", "rmat", "mesh"])
    n = _log(rng, 300, 1 << 23)
    if kind == "mesh":
        side = max(8, int(math.sqrt(n)))
        n = side * side
    c |= {"kind": kind, "n": n, "ncols": n, "d": 5 if kind == "mesh" else rng.choice([2, 4, 8, 16, 24, 32])}
    if kind == "rmat":
        c["symm"] = rng.random() < 0.6
    if kind == "er" and rng.random() < 0.5:  # rectangular
        c["ncols"] = _log(rng, max(64, n // 16), min(1 << 24, n * 4))
    if op == "permute":
        c["perm"] = rng.choice(["sym", "degree", "pair", "rows", "cols"] if c["ncols"] == n else ["pair", "rows", "cols"])
        return c
    c["sel"] = rng.choice(["random", "random", "sorted", "range"])
    if op == "extract":
        c |= {"nI": _log(rng, max(1, n // 64), n), "nJ": _log(rng, max(1, c["ncols"] // 64), c["ncols"])}
        if c["ncols"] == n and rng.random() < 0.3:
            c |= {"sel": "same", "nJ": c["nI"]}
        return c
    c |= {"nI": _log(rng, max(1, n // 256), n // 4), "nJ": _log(rng, max(8, c["ncols"] // 256), c["ncols"] // 4),
          "bd": rng.choice([2, 4, 8]), "mode": rng.choice(["replace", "replace", "second", "plus"])}
    return c


# ---- sizes, from the case alone -----------------------------------------------------------
def _rmat_scale(n):
    return max(1, (n - 1).bit_length())


def _rmat_expected(n, d, symm):
    """Expected number of distinct entries among ``d << scale`` R-MAT edges cut to n x n.

    A cell whose two indices agree in i zero bits and l one bits (and differ in the rest)
    is drawn with probability a^i b^(scale-i-l) d^l (b = c), so the cells are counted by
    (i, l), bit by bit from the top, keeping track of whether an index still equals n's
    leading bits and whether the two indices are still equal."""
    scale = _rmat_scale(n)
    full = n == 1 << scale
    states = {(not full, not full, True): {(0, 0): 1}}  # (row bound tight, column bound tight, diagonal)
    for bit in range(scale - 1, -1, -1):
        nb = (n >> bit) & 1 if not full else 1
        new = {}
        for (ts, td, dg), cells in states.items():
            for x in (0, 1):
                for y in (0, 1):
                    if (ts and x > nb) or (td and y > nb):
                        continue
                    to = new.setdefault((ts and x == nb, td and y == nb, dg and x == y), {})
                    for (i, l), k in cells.items():
                        at = (i + (x == 0 and y == 0), l + (x == 1 and y == 1))
                        to[at] = to.get(at, 0) + k
        states = new
    edges, total = d << scale, 0.0
    for (ts, td, dg), cells in states.items():
        if ts or td:
            continue  # equal to n: one past the last index
        for (i, l), k in cells.items():
            rate = edges * _RMAT[0] ** i * _RMAT[1] ** (scale - i - l) * _RMAT[3] ** l
            total += k * -math.expm1(-rate * (2 if symm and not dg else 1))
    return total


def _below(x, least=0):
    """A count that a random one with mean x seldom falls below."""
    return max(least, int(x - 4 * math.sqrt(x)))


def _entries(c, n=None, ncols=None):
    """Stored entries of a matrix of the case (of n rows, where the case has several)."""
    n = c["n"] if n is None else n
    ncols = c.get("ncols", n) if ncols is None else ncols
    if c["kind"] == "mesh":
        return _below(5 * n - 4 * math.isqrt(n))
    if c["kind"] == "er":
        return _below(n * ncols * -math.expm1(c["d"] * math.log1p(-1 / ncols)))
    return _below(_rmat_expected(n, c["d"], c["symm"]))


def _inside(c):
    """Stored entries of A(I, J)."""
    nI, nJ, nnz = c["nI"], c["nJ"], _entries(c)
    x = nnz / c["n"] * nI / c["ncols"] * nJ
    if c["kind"] == "mesh":  # about the diagonal
        x = 4 / 5 * x + nI if c["sel"] == "same" else x if c["sel"] != "range" else x / 4
    return min(_below(x, min(8, (nI * nJ + 1) // 2)), nnz, (9 * nI * nJ + 9) // 10)


def _b_entries(c):
    """Stored entries of B: (where A stores one, elsewhere) for the union modes, all for replace."""
    nI, nJ = c["nI"], c["nJ"]
    all_ = max(1, int(0.99 * nI * nJ * -math.expm1(c["bd"] * math.log1p(-1 / nJ) if nJ > 1 else -1)))
    if c["mode"] == "replace":
        return 0, all_
    over = min(_inside(c), all_ // 2)
    return over, min(all_ - over, (nI * nJ - _inside(c) + 1) // 2)


def _log_sizes(lo, hi, count, rng):
    """``count`` sizes spread evenly over the logarithm of [lo, hi], in a shuffled order."""
    x = [int(round(math.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * (k + 0.5) / count))) for k in range(count)]
    rng.shuffle(x)
    return x


def _batch(c):
    """Rows of the matrices, and per request its matrix and (batch-extract) |I| and |J|."""
    rng = random.Random(repr(sorted((k, v) for k, v in c.items() if k != "name")))
    rows = _log_sizes(1024, c["n"], c["nmats"], rng)
    which = [k % c["nmats"] for k in range(c["nreq"])]
    rng.shuffle(which)
    if c["op"] == "batch-permute":
        return rows, [(k, rows[k], rows[k]) for k in which]
    ni, nj = _log_sizes(16, c["most"], c["nreq"], rng), _log_sizes(16, c["most"], c["nreq"], rng)
    return rows, [(k, min(a, rows[k]), min(b, rows[k])) for k, a, b in zip(which, ni, nj)]


def _batch_kept(c):
    rows, reqs = _batch(c)
    nnz = [_entries(c, n) for n in rows]
    return sum(nnz[k] * (a / rows[k]) * (b / rows[k]) for k, a, b in reqs)


# ---- inputs ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _unique(keys):
    keys = keys.sort().values
    keep = torch.ones_like(keys, dtype=torch.bool)
    keep[1:] = keys[1:] != keys[:-1]
    return keys[keep]


def _has(keys, x):
    """Whether each of x is among the sorted keys."""
    if keys.numel() == 0:
        return torch.zeros_like(x, dtype=torch.bool)
    return keys[torch.searchsorted(keys, x).clamp_(max=keys.numel() - 1)] == x


def _some(n, k, g):
    """k distinct positions below n."""
    if 4 * k > n:
        return torch.randperm(n, device=DEV, generator=g)[:k]
    x = torch.empty(0, dtype=torch.int64, device=DEV)
    while x.numel() < k:
        x = _unique(torch.cat([x, torch.randint(0, n, (k + k // 4 + 16,), device=DEV, generator=g)]))
    return x[torch.randperm(x.numel(), device=DEV, generator=g)[:k]]


def _drop(keys, which, k, g):
    """The keys without k of those at the positions `which` (None: of all)."""
    if k <= 0:
        return keys
    keep = torch.ones_like(keys, dtype=torch.bool)
    at = _some(keys.numel() if which is None else which.numel(), k, g)
    keep[at if which is None else which[at]] = False
    return keys[keep]


def _fresh(keys, k, sample):
    """k keys from sample(count) that are not among the sorted keys."""
    new = torch.empty(0, dtype=torch.int64, device=DEV)
    while new.numel() < k:
        x = _unique(torch.cat([new, sample(2 * k + 64)]))
        new = x[~_has(keys, x)]
    return new


def _add(keys, k, sample, g):
    if k <= 0:
        return keys
    new = _fresh(keys, k, sample)
    new = new[torch.randperm(new.numel(), device=DEV, generator=g)[:k]]
    return torch.cat([keys, new]).sort().values


def _er_keys(m, n, d, g, chunk=1 << 22):
    """``d`` uniform columns a row, repeats merged."""
    out = []
    for r0 in range(0, m, chunk):
        k = min(chunk, m - r0)
        x = torch.randint(0, n, (k, d), dtype=torch.int32, device=DEV, generator=g).sort(1).values
        keep = torch.ones_like(x, dtype=torch.bool)
        keep[:, 1:] = x[:, 1:] != x[:, :-1]
        out.append((x + torch.arange(r0, r0 + k, device=DEV)[:, None] * n)[keep])
    return torch.cat(out) if len(out) > 1 else out[0]


def _rmat_keys(n, d, symm, g, chunk=1 << 27):
    """``d`` edges a vertex of an R-MAT graph, cut to its leading n vertices, repeats merged."""
    scale = _rmat_scale(n)
    a, ab, abc = _RMAT[0], _RMAT[0] + _RMAT[1], _RMAT[0] + _RMAT[1] + _RMAT[2]
    parts, edges = [], d << scale
    for e0 in range(0, edges, chunk):
        k = min(chunk, edges - e0)
        src = torch.zeros(k, dtype=torch.int32, device=DEV)
        dst = torch.zeros_like(src)
        for _ in range(scale):
            u = torch.rand(k, device=DEV, generator=g)
            src.mul_(2).add_(u >= ab)
            dst.mul_(2).add_(((u >= a) & (u < ab)) | (u >= abc))
        if n < 1 << scale:
            keep = (src < n) & (dst < n)
            src, dst = src[keep], dst[keep]
        src, dst = src.to(torch.int64), dst.to(torch.int64)
        parts.append(src * n + dst)
        if symm:
            parts.append(dst * n + src)
    del src, dst
    keys = torch.cat(parts) if len(parts) > 1 else parts[0]
    del parts
    return _unique(keys)


def _mesh_keys(n):
    side = math.isqrt(n)
    v = torch.arange(n, dtype=torch.int64, device=DEV)
    r, k = v // side, v % side
    cand = torch.stack([v - side, v - 1, v, v + 1, v + side], 1)
    ok = torch.stack([r > 0, k > 0, torch.ones_like(r, dtype=torch.bool), k < side - 1, r < side - 1], 1)
    return (cand + v[:, None] * n)[ok]


def _keys(c, g, n=None):
    """Sorted places (row * ncols + column) of about the case's number of entries."""
    n = c["n"] if n is None else n
    if c["kind"] == "er":
        return _er_keys(n, c["ncols"], c["d"], g)
    return _mesh_keys(n) if c["kind"] == "mesh" else _rmat_keys(n, c["d"], c["symm"], g)


def _to_count(keys, count, m, n, g):
    """`keys` with as many dropped or added as make `count`."""
    keys = _drop(keys, None, keys.numel() - count, g)
    return _add(keys, count - keys.numel(), lambda k: torch.randint(0, m * n, (k,), device=DEV, generator=g), g)


def _csr(keys, m, n, c, g):
    rowptr = torch.searchsorted(keys, torch.arange(m + 1, dtype=torch.int64, device=DEV) * n)
    val = torch.rand(keys.numel(), dtype=_FLT[c["vt"]], device=DEV, generator=g)
    if c["vt"] == 64:
        val = val.mul_(2.0).sub_(1.0)
    return CSR(m, n, rowptr.to(_INT[c["rp"]]), (keys % n).to(_INT[c["ci"]]), val)


def _perm(n, c, g):
    return torch.randperm(n, device=DEV, generator=g).to(_INT[c["ix"]])


def _select(n, k, how, g):
    """k of n indices: in random order, ascending, or consecutive."""
    if how == "range":
        lo = int(torch.randint(0, n - k + 1, (1,), device=DEV, generator=g))
        return torch.arange(lo, lo + k, device=DEV)
    x = torch.randperm(n, device=DEV, generator=g)[:k]
    return x.sort().values if how == "sorted" else x


def _member(x, n):
    m = torch.zeros(n, dtype=torch.bool, device=DEV)
    m[x] = True
    return m


def _with_region(keys, c, I, J, g):
    """`keys` with exactly ``_inside`` entries at rows of I and columns of J (and, for an
    assignment, ``_entries`` in all); and which are inside."""
    m, n = c["n"], c["ncols"]
    mi, mj = _member(I, m), _member(J, n)

    def inside(x):
        return mi[x // n] & mj[x % n]

    def pairs(k):
        r = I[torch.randint(0, I.numel(), (k,), device=DEV, generator=g)]
        return r * n + J[torch.randint(0, J.numel(), (k,), device=DEV, generator=g)]

    def elsewhere(k):
        x = torch.randint(0, m * n, (k,), device=DEV, generator=g)
        return x[~inside(x)]

    here, there = _inside(c), _entries(c) - _inside(c)
    at = inside(keys).nonzero()[:, 0]
    keys = _add(_drop(keys, at, at.numel() - here, g), here - at.numel(), pairs, g)
    if c["op"] != "extract":  # whose result holds none of the others
        at = (~inside(keys)).nonzero()[:, 0]
        keys = _add(_drop(keys, at, at.numel() - there, g), there - at.numel(), elsewhere, g)
    return keys, inside


def _patch(keys, inside, c, I, J, g):
    """B of an assignment at (I, J)."""
    nI, nJ = c["nI"], c["nJ"]
    over, new = _b_entries(c)
    if c["mode"] == "replace":
        return _csr(_to_count(_er_keys(nI, nJ, c["bd"], g), new, nI, nJ, g), nI, nJ, c, g)
    # the union modes: `over` of A's entries in the region and `new` places beside them
    n = c["ncols"]
    ri, rj = _inverse(I, c["n"]), _inverse(J, n)
    at = keys[inside(keys)]
    at = (ri[at // n] * nJ + rj[at % n]).sort().values
    some = at[_some(at.numel(), over, g)].sort().values
    fresh = _fresh(at, new, lambda k: torch.randint(0, nI * nJ, (k,), device=DEV, generator=g))
    fresh = fresh[torch.randperm(fresh.numel(), device=DEV, generator=g)[:new]]
    return _csr(torch.cat([some, fresh]).sort().values, nI, nJ, c, g)


def prepare(case, seed):
    c, g = case, _gen(seed)
    s = {"c": c, "ctx": _context()}
    if c["op"].startswith("batch"):
        # resident matrices of uneven sizes, each with a pool of random indices that its
        # requests' vectors are cut from
        rows, reqs = _batch(c)
        s["mats"] = [_csr(_to_count(_keys(c, g, n), _entries(c, n), n, n, g), n, n, c, g) for n in rows]
        if c["op"] == "batch-permute":
            s["reqs"] = [(k, p, p) for k, n, _ in reqs for p in (_perm(n, c, g),)]
            return s
        pools = [_perm(n, c, g) for n in rows]
        starts = torch.rand(len(reqs), 2, device=DEV, generator=g, dtype=torch.float64).tolist()
        s["reqs"] = []
        for (k, a, b), (x, y) in zip(reqs, starts):
            x, y = int(x * (rows[k] - a + 1)), int(y * (rows[k] - b + 1))
            s["reqs"].append((k, pools[k][x:x + a], pools[k][y:y + b]))
        s["batch"] = ExtractBatch(s["ctx"], s["mats"], s["reqs"])
        # an output buffer of the size that a server holds ready for such a round
        room = 2 * int(_batch_kept(c)) + (1 << 16)
        if s["batch"].nnz > room:
            raise ValueError("the round's output does not fit its buffer")
        like = s["mats"][0]
        s["out"] = CSR(s["batch"].rows, s["batch"].ncols,
                       torch.zeros(s["batch"].rows + 1, dtype=torch.int64, device=DEV),
                       torch.zeros(room, dtype=like.colidx.dtype, device=DEV),
                       torch.zeros(room, dtype=like.values.dtype, device=DEV))
        return s
    m, n = c["n"], c["ncols"]
    keys = _keys(c, g)
    if c["op"] == "permute":
        A = s["A"] = _csr(_to_count(keys, _entries(c), m, n, g), m, n, c, g)
        s["p"] = s["q"] = None
        if c["perm"] == "degree":
            deg = A.rowptr[1:] - A.rowptr[:-1]
            s["p"] = s["q"] = deg.sort(descending=True, stable=True).indices.to(_INT[c["ix"]])
        if c["perm"] in ("sym", "pair", "rows"):
            s["p"] = _perm(m, c, g)
        if c["perm"] in ("pair", "cols"):
            s["q"] = _perm(n, c, g)
        if c["perm"] == "sym":
            s["q"] = s["p"]
        return s
    same = c["sel"] == "same"
    I = _select(m, c["nI"], "random" if same else c["sel"], g)
    J = I if same else _select(n, c["nJ"], c["sel"], g)
    keys, inside = _with_region(keys, c, I, J, g)
    s["A"] = _csr(keys, m, n, c, g)
    if c["op"] != "extract":
        s["B"] = _patch(keys, inside, c, I, J, g)
    s["I"] = I.to(_INT[c["ix"]])
    s["J"] = s["I"] if same else J.to(_INT[c["ix"]])
    if c["op"] == "update":
        s["p"] = _perm(m, c, g)
        s["q"] = s["p"] if m == n else _perm(n, c, g)
    return s


# ---- one pass --------------------------------------------------------------------------
def _arrays(M):
    return {"rowptr": M.rowptr, "colidx": M.colidx, "values": M.values}


def run(state):
    s, c, ctx = state, state["c"], state["ctx"]
    if c["op"] == "permute":
        return _arrays(ctx.sp_permute(s["A"], s["p"], s["q"]))
    if c["op"] == "extract":
        return _arrays(ctx.sp_extract(s["A"], s["I"], s["J"]))
    if c["op"] == "assign":
        return _arrays(ctx.sp_assign(s["A"], s["I"], s["J"], s["B"], mode=_MODE[c["mode"]]))
    if c["op"] == "update":
        return _arrays(ctx.sp_assign_permute(s["A"], s["I"], s["J"], s["B"], s["p"], s["q"], mode=_MODE[c["mode"]]))
    if c["op"] == "batch-extract":
        s["batch"].run(s["out"])
        ctx.sync()
        return _arrays(s["out"])
    out, first = ctx.sp_permute_batch(s["mats"], s["reqs"])
    return _arrays(out) | {"first": torch.tensor(first)}


# ---- what a pass cannot do without -----------------------------------------------------
def work(case):
    """Each input read once and each output written once: all of the matrices for a
    permutation or an assignment; for an extraction the selected rows' row pointers and
    columns (of a consecutive J only the kept ones), and the values of what is kept."""
    c = case
    rp, ci, ix, vt = (c[k] // 8 for k in ("rp", "ci", "ix", "vt"))
    e = ci + vt
    if c["op"].startswith("batch"):
        rows, reqs = _batch(c)
        nnz = [_entries(c, n) for n in rows]
        if c["op"] == "batch-permute":
            return {"bytes": sum(2 * nnz[k] * e + n * (ix + rp + 8) for k, n, _ in reqs), "flops": 0}
        scanned = sum(nnz[k] * a / rows[k] for k, a, _ in reqs)
        return {"bytes": scanned * ci + _batch_kept(c) * (vt + e) + sum(a * (ix + 2 * rp + 8) + b * ix for _, a, b in reqs),
                "flops": 0}
    nnz, m, n = _entries(c), c["n"], c["ncols"]
    if c["op"] == "permute":
        index = {"pair": m + n, "rows": m, "cols": n}.get(c["perm"], m) * ix  # sym, degree: one vector
        return {"bytes": 2 * nnz * e + 2 * m * rp + index, "flops": 0}
    nI, nJ, kept = c["nI"], c["nJ"], _inside(c)
    if c["op"] == "extract":
        scanned = kept if c["sel"] == "range" else nnz * nI / m
        return {"bytes": scanned * ci + kept * (vt + e) + nI * (ix + 3 * rp) + nJ * ix, "flops": 0}
    over, new = _b_entries(c)
    out = nnz + new - (kept if c["mode"] == "replace" else 0)
    index = nI * (ix + rp) + nJ * ix + ((m if m == n else m + n) * ix if c["op"] == "update" else 0)
    return {"bytes": (nnz + over + new + out) * e + 2 * m * rp + index,
            "flops": over if c["mode"] == "plus" else 0}


# ---- 64-bit values ---------------------------------------------------------------------
def _triplets(A):
    lens = (A.rowptr[1:] - A.rowptr[:-1]).long()
    return torch.repeat_interleave(torch.arange(A.nrows, device=DEV), lens), A.colidx.long(), A.values.double()


def _inverse(x, n):
    inv = torch.full((n,), -1, dtype=torch.int64, device=DEV)
    inv[x.long()] = torch.arange(x.numel(), device=DEV)
    return inv


def _by_place(r, c, v, n):
    return v[torch.sort(r * n + c).indices]


def _permuted(r, c, v, m, n, p, q):
    r = r if p is None else _inverse(p, m)[r]
    c = c if q is None else _inverse(q, n)[c]
    return _by_place(r, c, v, n)


def _extracted(A, I, J):
    r, c, v = _triplets(A)
    r, c = _inverse(I, A.nrows)[r], _inverse(J, A.ncols)[c]
    keep = (r >= 0) & (c >= 0)
    return _by_place(r[keep], c[keep], v[keep], max(1, J.numel()))


def exact(case, seed):
    s, c = prepare(case, seed), case
    if c["op"] == "batch-extract":
        v = torch.zeros(s["out"].nnz, dtype=torch.float64, device=DEV)
        kept = torch.cat([_extracted(s["mats"][k], I, J) for k, I, J in s["reqs"]])
        v[:kept.numel()] = kept
    elif c["op"] == "batch-permute":
        tri = [_triplets(A) for A in s["mats"]]
        v = torch.cat([_permuted(*tri[k], s["mats"][k].nrows, s["mats"][k].ncols, p, q) for k, p, q in s["reqs"]])
        return {"rowptr": None, "colidx": None, "values": v, "first": None}
    elif c["op"] == "permute":
        v = _permuted(*_triplets(s["A"]), s["A"].nrows, s["A"].ncols, s["p"], s["q"])
    elif c["op"] == "extract":
        v = _extracted(s["A"], s["I"], s["J"])
    else:
        m, n = s["A"].nrows, s["A"].ncols
        r, k, v = _triplets(s["A"])
        br, bk, bv = _triplets(s["B"])
        if c["mode"] == "replace":
            keep = (_inverse(s["I"], m)[r] < 0) | (_inverse(s["J"], n)[k] < 0)
            r, k, v = r[keep], k[keep], v[keep]
        # B's entries behind A's: of two in one place, the sum or the later one
        key = torch.cat([r * n + k, s["I"].long()[br] * n + s["J"].long()[bk]])
        v = torch.cat([v, bv])
        key, order = torch.sort(key, stable=True)
        v = v[order]
        same = key[1:] == key[:-1]
        if c["mode"] == "plus":
            v[:-1][same] += v[1:][same]
            keep = torch.cat([torch.ones(1, dtype=torch.bool, device=DEV), ~same])
        else:
            keep = torch.cat([~same, torch.ones(1, dtype=torch.bool, device=DEV)])
        key, v = key[keep], v[keep]
        if c["op"] == "update":
            v = _permuted(key // n, key % n, v, m, n, s["p"], s["q"])
    return {"rowptr": None, "colidx": None, "values": v}
