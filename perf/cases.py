"""The work that users of this library have it do, as measurable cases.

A case is one call of a public entry point (or, for the request server, one
wave of requests) on a seeded synthetic matrix of the structures that the
repository's workloads use: uniform random sparse, 2D 5-point and 3D 27-point
stencils, banded and R-MAT power-law graphs, weights log-normal and
transformed per column, a planted perfect matching.  Inputs are made on the
GPU from the seed alone.  Contexts are kept per process, one per set of
options, as a program that solves many matrices keeps its context.

`exact` restates every path in plain torch: 64-bit integers and doubles,
without this repository's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1801_09809_gb300 import awpm

DEV = "cuda"
BIG = 1 << 62


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one pre-pivoting matrix of 2,000 rows, where
        # launches and the host path count
        {"name": "improve_random_n2000", "op": "improve", "kind": "random", "n": 2000, "deg": 8},
        # ordinary large matrices: a 2D discretisation of a million unknowns,
        # few passes, five entries per column
        {"name": "improve_grid5_1000", "op": "improve", "kind": "grid5", "side": 1000},
        # a 3D discretisation, 27 entries per column, many passes
        {"name": "improve_grid27_96", "op": "improve", "kind": "grid27", "side": 96},
        # the largest single matrix: power-law degrees, 69 M entries, far
        # larger than L2
        {"name": "improve_rmat_s22", "op": "improve", "kind": "rmat", "n": 1 << 22, "deg": 16},
        # the other selection rule (greedy D(S)), a 3D discretisation of
        # ordinary size
        {"name": "improve_select_grid27_64", "op": "improve", "kind": "grid27", "side": 64,
         "select": 1},
        # thousands of small matrices in one call (block-diagonal systems,
        # ensembles)
        {"name": "batch_4096", "op": "batch", "count": 4096, "lo": 200, "hi": 20000},
        # a wave of requests of all sizes through the request server, inputs
        # in pinned host memory
        {"name": "serve_32", "op": "serve", "count": 32, "lo": 1000, "hi": 1000000},
        # the whole pipeline from no matching: greedy, maximum matching,
        # 4-cycle phase
        {"name": "pipeline_rmat_s22", "op": "pipeline", "kind": "rmat", "n": 1 << 22, "deg": 16},
        # the greedy maximal matching alone, a million columns
        {"name": "greedy_random_1m", "op": "greedy", "kind": "random", "n": 1000000, "deg": 16},
        # completing a partial matching (5 % of the columns unmatched)
        {"name": "mcm_random_250k", "op": "mcm", "kind": "random", "n": 250000, "deg": 6},
        # weights from the values of the largest matrix (logarithms)
        {"name": "weights_log_rmat_s22", "op": "weights", "kind": "rmat", "n": 1 << 22, "deg": 16,
         "mode": 1},
        # one search without allocations for a host framework, an odd size
        {"name": "noalloc_banded_100003", "op": "noalloc", "kind": "banded", "n": 100003,
         "deg": 15},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["improve", "improve", "improve", "batch", "serve", "pipeline", "greedy",
                     "mcm", "weights", "search", "noalloc"])
    if op == "batch":
        return {"op": op, "count": _log_int(rng, 4, 2048), "lo": rng.randint(50, 400),
                "hi": rng.randint(4000, 20000)}
    if op == "serve":
        return {"op": op, "count": rng.randint(4, 24), "lo": rng.randint(300, 3000),
                "hi": rng.randint(100000, 900000)}
    kind = rng.choice(["random", "grid5", "grid27", "banded", "rmat"])
    cap = {"improve": 1 << 21, "search": 1 << 21, "weights": 1 << 21, "greedy": 1 << 20,
           "pipeline": 1 << 19, "mcm": 1 << 18, "noalloc": 130000}[op]
    if op in ("pipeline", "mcm") and kind in ("banded", "grid5", "grid27"):
        cap = 20000  # long augmenting paths: many search levels for the size
    n = _log_int(rng, 300, cap)
    case = {"op": op, "kind": kind}
    if kind == "grid5":
        case["side"] = max(2, int(math.sqrt(n)))
    elif kind == "grid27":
        case["side"] = min(80, max(3, int(round(n ** (1.0 / 3.0)))))
    else:
        case["n"] = n
        case["deg"] = rng.choice(range(3, 16, 2)) if kind == "banded" else rng.randint(4, 27)
    if op == "improve":
        case["select"] = rng.choice([0, 0, 0, 1])
        case["lookup"] = rng.choice([0, 0, 0, 0, 1, 2, 3])
    if op == "weights":
        case["mode"] = rng.randint(0, 1)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _block_perm(block, g):
    """A random permutation inside every block (block: block number of each index,
    ascending)."""
    x = torch.rand(block.numel(), generator=g, device=DEV, dtype=torch.float64)
    return torch.argsort(block.double() + x * 0.999, stable=True)


def _csc(N, rows, cols, z, diag, g):
    """CSC arrays of the entries (rows, cols) and the planted pairs (diag[j], j);
    weights from `z` (a function of the number of entries), transformed per
    column to log magnitudes with maximum 0."""
    ids = torch.arange(N, device=DEV)
    key = torch.unique(torch.cat([cols * N + rows, ids * N + diag]))
    col = key // N
    row = key - col * N
    colptr = torch.zeros(N + 1, device=DEV, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(col, minlength=N), 0)
    x = z(row, col, key.numel(), g)
    top = torch.full((N,), -math.inf, device=DEV, dtype=torch.float64)
    top.scatter_reduce_(0, col, x, "amax")
    return (colptr.int(), row.int(), x - top[col], diag.int().contiguous())


def _lognormal(row, col, m, g):
    return torch.randn(m, generator=g, device=DEV, dtype=torch.float64)


def _blocks(kinds, ns, params, g):
    """One block-diagonal union of random ('random', degree), 2D 5-point ('grid5',
    side), 3D 27-point ('grid27', side) and banded ('banded', width) matrices."""
    ns_t = torch.tensor(ns, device=DEV)
    off = torch.zeros(len(ns) + 1, device=DEV, dtype=torch.int64)
    off[1:] = torch.cumsum(ns_t, 0)
    N = int(sum(ns))
    slots = [p if k in ("random", "banded") else 5 if k == "grid5" else 27
             for k, p in zip(kinds, params)]
    block = torch.repeat_interleave(torch.arange(len(ns), device=DEV), ns_t)
    code = torch.tensor([("random", "grid5", "grid27", "banded").index(k) for k in kinds],
                        device=DEV)[block]
    par = torch.tensor(params, device=DEV)[block]
    per = torch.tensor(slots, device=DEV)[block]
    col = torch.repeat_interleave(torch.arange(N, device=DEV), per)
    first = torch.cumsum(per, 0) - per
    slot = torch.arange(col.numel(), device=DEV) - first[col]
    b, c, p = block[col], code[col], par[col]
    n, lj = ns_t[b], col - off[b]
    u = torch.rand(col.numel(), generator=g, device=DEV, dtype=torch.float64)
    row = (u * n).long().clamp_(max=0x7FFFFFFF)
    row = torch.minimum(row, n - 1)
    ok = torch.ones_like(col, dtype=torch.bool)
    # 5-point: offsets (0,0) (1,0) (-1,0) (0,1) (0,-1)
    x, y = lj % p, lj // p
    dx = (slot == 1).long() - (slot == 2).long()
    dy = (slot == 3).long() - (slot == 4).long()
    inside = (x + dx >= 0) & (x + dx < p) & (y + dy >= 0) & (y + dy < p)
    is5 = c == 1
    row = torch.where(is5, (y + dy) * p + x + dx, row)
    ok = torch.where(is5, inside, ok)
    # 27-point
    x, y, zc = lj % p, (lj // p) % p, lj // (p * p)
    dx, dy, dz = slot % 3 - 1, (slot // 3) % 3 - 1, slot // 9 - 1
    inside = ((x + dx >= 0) & (x + dx < p) & (y + dy >= 0) & (y + dy < p) &
              (zc + dz >= 0) & (zc + dz < p))
    is27 = c == 2
    row = torch.where(is27, ((zc + dz) * p + y + dy) * p + x + dx, row)
    ok = torch.where(is27, inside, ok)
    # banded
    d = slot - (p - 1) // 2
    isb = c == 3
    row = torch.where(isb, lj + d, row)
    ok = torch.where(isb, (lj + d >= 0) & (lj + d < n), ok)
    rows, cols = (row + off[b])[ok], col[ok]
    # rows permuted inside every block; columns too for the 3D stencils
    pi = _block_perm(block, g)
    sg = torch.where(code == 2, _block_perm(block, g), torch.arange(N, device=DEV))
    diag = torch.empty(N, device=DEV, dtype=torch.int64)
    diag[sg] = pi
    return N, off, pi[rows], sg[cols], diag


def _rmat(n, deg, g):
    m = n * deg
    scale = max(1, (n - 1).bit_length())
    r = torch.zeros(m, device=DEV, dtype=torch.int32)
    c = torch.zeros(m, device=DEV, dtype=torch.int32)
    for _ in range(scale):
        u = torch.rand(m, generator=g, device=DEV)
        r.mul_(2).add_(u >= 0.76)
        c.mul_(2).add_(((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    ok = (r < n) & (c < n)
    zero = torch.zeros(n, device=DEV, dtype=torch.int64)
    pr, pc, pm = (_block_perm(zero, g) for _ in range(3))
    return pr[r[ok].long()], pc[c[ok].long()], pm


def _matrix(kind, size, param, seed):
    """(n, colptr, rowidx, weight, mate) of one matrix."""
    g = _gen(seed)
    if kind == "rmat":
        rows, cols, diag = _rmat(size, param, g)
        return (size, *_csc(size, rows, cols, _lognormal, diag, g))
    n = size ** 2 if kind == "grid5" else size ** 3 if kind == "grid27" else size
    N, _, rows, cols, diag = _blocks([kind], [n], [param], g)
    z = _lognormal
    if kind == "grid5":
        # diagonal |a| ~ U[0.5, 1.5], off-diagonal a ~ N(0, 1)
        def z(row, col, m, g):
            on = torch.rand(m, generator=g, device=DEV, dtype=torch.float64) + 0.5
            out = torch.randn(m, generator=g, device=DEV, dtype=torch.float64).abs()
            return torch.log(torch.where(row == diag[col], on, out.clamp_(min=1e-300)))
    return (N, *_csc(N, rows, cols, z, diag, g))


def _single(case):
    kind = case["kind"]
    if kind in ("grid5", "grid27"):
        return kind, case["side"], case["side"]
    return kind, case["n"], min(case["deg"], case["n"])


def _quantiles(case):
    """Sizes log-uniform over [lo, hi], one per quantile."""
    k, lo, hi = case["count"], case["lo"], case["hi"]
    return [int(round(lo * (hi / lo) ** ((x + 0.5) / k))) for x in range(k)]


def _batch_spec(case):
    kinds, ns, params = [], [], []
    for x, n in enumerate(_quantiles(case)):
        kind = ("random", "grid5", "banded")[x % 3]
        if kind == "grid5":
            p = max(2, int(round(math.sqrt(n))))
            n = p * p
        else:
            p = 4 + (x * 5) % 13 if kind == "random" else 3 + 2 * ((x * 3) % 7)
        kinds.append(kind)
        ns.append(n)
        params.append(p)
    order = sorted(range(len(ns)), key=lambda x: (x * 2654435761) % 4294967296)
    return [kinds[x] for x in order], [ns[x] for x in order], [params[x] for x in order]


def _serve_spec(case):
    out = []
    for x, n in enumerate(_quantiles(case)):
        kind = ("random", "grid5", "grid27", "rmat")[x % 4]
        if kind == "grid5":
            size = param = max(2, int(round(math.sqrt(n))))
        elif kind == "grid27":
            size = param = max(2, int(round(n ** (1.0 / 3.0))))
        else:
            size, param = n, 4 + (x * 7) % 24
        out.append((kind, size, param))
    return sorted(out, key=lambda s: (s[1] * 2654435761 + s[2]) % 4294967296)


def _room(case):
    kind, size, param = _single(case)
    n = size ** 2 if kind == "grid5" else size ** 3 if kind == "grid27" else size
    per = {"grid5": 5, "grid27": 27, "banded": param}.get(kind, param + 1)
    return n * per


_contexts = {}


def _context(**options):
    key = tuple(sorted(options.items()))
    if key not in _contexts:
        _contexts[key] = awpm.awpm_create(device=torch.cuda.current_device(), **options)
    return _contexts[key]


def prepare(case, seed):
    op = case["op"]
    st = {"op": op}
    if op == "batch":
        g = _gen(seed)
        N, off, rows, cols, diag = _blocks(*_batch_spec(case), g)
        colptr, rowidx, weight, mate = _csc(N, rows, cols, _lognormal, diag, g)
        st.update(n=N, off=off.int(), colptr=colptr, rowidx=rowidx, weight=weight, mate=mate,
                  out=torch.empty_like(mate), count=case["count"], ctx=_context())
        return st
    if op == "serve":
        reqs = []
        for x, (kind, size, param) in enumerate(_serve_spec(case)):
            n, *arrays = _matrix(kind, size, param, seed * 1000003 + x)
            pinned = []
            for a in arrays:
                h = torch.empty(a.shape, dtype=a.dtype, pin_memory=True)
                h.copy_(a)
                pinned.append(h)
            reqs.append((n, pinned, torch.empty(n, dtype=torch.int32, pin_memory=True)))
        st.update(reqs=reqs, ctx=_context(slots=4, mem_budget_bytes=100_000_000_000))
        return st
    n, colptr, rowidx, weight, mate = _matrix(*_single(case), seed)
    st.update(n=n, colptr=colptr, rowidx=rowidx, weight=weight, mate=mate,
              out=torch.empty_like(mate))
    if op == "improve":
        st["ctx"] = _context(lookup=case.get("lookup", 0), select=case.get("select", 0))
    elif op != "noalloc":
        st["ctx"] = _context()
    if op == "mcm":
        u = torch.rand(n, generator=_gen(seed + 77), device=DEV)
        st["mate"] = torch.where(u < 0.05, torch.full_like(mate, -1), mate)
    if op == "weights":
        # matrix values: log-normal magnitudes of either sign
        g = _gen(seed + 78)
        a = torch.exp(torch.randn(weight.numel(), generator=g, device=DEV, dtype=torch.float64))
        s = torch.rand(weight.numel(), generator=g, device=DEV) < 0.5
        st["weight"] = torch.where(s, -a, a)
        st["mode"] = case["mode"]
        # room for the entries of any seed's matrix; what is past them stays 0
        st["wout"] = torch.zeros(_room(case), device=DEV, dtype=torch.float64)
    if op in ("search", "noalloc"):
        st["gain"] = torch.empty(n, device=DEV, dtype=torch.float64)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _phase_out(mate, s):
    return {"mate": mate,
            "counts": np.array([s["iterations"], s["converged"], s["cycles_applied"],
                                s["edge_checks"], s["candidates"], s["closing_found"],
                                s["positive"]], dtype=np.int64),
            "weights": np.array([s["weight_in"], s["weight_out"]])}


def run(st):
    op = st["op"]
    if op == "serve":
        ctx = st["ctx"]
        tickets = [awpm.awpm_submit(ctx, n, *a, out, nnz=a[1].numel()) for n, a, out in st["reqs"]]
        stats = [awpm.awpm_wait(ctx, t) for t in tickets]
        return {"mates": [out for _, _, out in st["reqs"]][:30],
                "counts": np.array([[s["iterations"], s["cycles_applied"], s["candidates"],
                                     s["closing_found"], s["positive"]] for s in stats],
                                   dtype=np.int64),
                "weights": np.array([[s["weight_in"], s["weight_out"]] for s in stats])}
    n, cp, ri, w = st["n"], st["colptr"], st["rowidx"], st["weight"]
    if op == "improve":
        return _phase_out(st["out"], awpm.awpm_improve_ctx(st["ctx"], n, cp, ri, w, st["mate"],
                                                           st["out"]))
    if op == "pipeline":
        return _phase_out(st["out"], awpm.awpm_improve_ctx(st["ctx"], n, cp, ri, w, None,
                                                           st["out"]))
    if op == "batch":
        s, _ = awpm.awpm_improve_batch(st["ctx"], st["count"], st["off"], cp, ri, w, st["mate"],
                                       st["out"], per_matrix=False)
        return {"mate": st["out"],
                "counts": np.array([s["iterations"], s["converged"], s["cycles_applied"],
                                    s["edge_checks"], s["candidates"], s["closing_found"],
                                    s["positive"]], dtype=np.int64),
                "weights": np.array([s["weight_in"], s["weight_out"]])}
    if op == "greedy":
        s = awpm.awpm_greedy(st["ctx"], n, cp, ri, w, st["out"])
        return {"mate": st["out"], "counts": np.array([s["rounds"], s["cardinality"]]),
                "weights": np.array([s["weight"]])}
    if op == "mcm":
        st["out"].copy_(st["mate"])
        s = awpm.awpm_mcm(st["ctx"], n, cp, ri, w, st["out"])
        return {"mate": st["out"], "counts": np.array([s["phases"], s["cardinality"],
                                                       s["levels"]])}
    if op == "weights":
        awpm.awpm_weights(st["ctx"], n, cp, ri, w, st["mode"], st["wout"])
        return {"weight": st["wout"]}
    if op == "search":
        s = awpm.awpm_search(st["ctx"], n, cp, ri, w, st["mate"], st["gain"], st["out"])
    else:
        s = awpm.awpm_search_noalloc(n, cp, ri, w, st["mate"], st["gain"], st["out"])
    return {"gain": st["gain"], "row": st["out"],
            "counts": np.array([s["candidates"], s["closing_found"], s["positive"]],
                               dtype=np.int64)}


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------

def _size(kind, size, param):
    """(n, expected entries)."""
    if kind == "grid5":
        return size ** 2, 5 * size ** 2 - 4 * size
    if kind == "grid27":
        return size ** 3, (3 * size - 2) ** 3
    if kind == "banded":
        h = (param - 1) // 2
        return size, size * (2 * h + 1) - h * (h + 1)
    if kind == "random":
        # distinct rows among `param` draws and the planted one
        return size, int(size * size * (1 - (1 - 1 / size) ** (param + 1)))
    return size, size * param + size  # R-MAT, before duplicates leave


def work(case):
    op = case["op"]
    if op == "batch":
        parts = [_size(k, p if k == "grid5" else n, p) for k, n, p in zip(*_batch_spec(case))]
    elif op == "serve":
        parts = [_size(*s) for s in _serve_spec(case)]
    else:
        parts = [_size(*_single(case))]
    n, nnz = sum(p[0] for p in parts), sum(p[1] for p in parts)
    pattern = 4 * nnz + 4 * (n + 1)
    if op == "weights":
        return {"bytes": pattern + 16 * nnz, "flops": (3 if case["mode"] else 2) * nnz}
    if op in ("search", "noalloc"):
        return {"bytes": pattern + 8 * nnz + 16 * n, "flops": 3 * (nnz - n) // 2}
    return {"bytes": pattern + 8 * nnz + 8 * n, "flops": 3 * (nnz - n) // 2}


def tolerance(case):
    op = case["op"]
    if op in ("search", "noalloc"):
        return "exact"  # one fixed order of three FP64 additions
    if op == "mcm":
        return "exact"  # whole numbers
    if op == "weights":
        # divisions and maxima are exact; the logarithm is good to an ulp
        return "exact" if case["mode"] == 0 else {"rel": 5e-16, "max": 1e-14}
    # matchings and counters are the same; the weights' sums may be taken in
    # another order (n additions of doubles of one sign)
    return {"rel": 1e-13}


# ---------------------------------------------------------------------------
# the same results in plain torch
# ---------------------------------------------------------------------------

class _M:
    def __init__(self, n, colptr, rowidx, weight):
        self.n, self.w = n, weight.to(DEV).double()
        self.ptr = colptr.to(DEV).long()
        self.row = rowidx.to(DEV).long()
        self.col = torch.repeat_interleave(torch.arange(n, device=DEV), self.ptr.diff())
        self.key = self.col * n + self.row


def _full(n, v, dt=torch.int64):
    return torch.full((n,), v, device=DEV, dtype=dt)


def _amax(n, at, v):
    return _full(n, -math.inf, torch.float64).scatter_reduce_(0, at, v, "amax")


def _amin(n, at, v):
    return _full(n, BIG).scatter_reduce_(0, at, v, "amin")


def _winners(m, mc, mr, wm):
    """Step-C winners: (j, p, q, gain)."""
    p = torch.nonzero(m.row > mc[m.col]).flatten()
    k = mr[m.row[p]] * m.n + mc[m.col[p]]
    q = torch.searchsorted(m.key, k).clamp_(max=m.key.numel() - 1)
    hit = m.key[q] == k
    p, q = p[hit], q[hit]
    j = m.col[p]
    g = ((m.w[p] + m.w[q]) - wm[mr[m.row[p]]]) - wm[j]
    pos = g > 0
    p, q, j, g = p[pos], q[pos], j[pos], g[pos]
    top = g == _amax(m.n, j, g)[j]
    p, q, j, g = p[top], q[top], j[top], g[top]
    low = p == _amin(m.n, j, p)[j]
    return j[low], p[low], q[low], g[low]


def _phase(m, mate, select):
    n = m.n
    ids = torch.arange(n, device=DEV)
    mc = mate.to(DEV).long().clone()
    mr = torch.empty_like(mc)
    mr[mc] = ids
    wm = m.w[torch.searchsorted(m.key, ids * n + mc)].clone()
    win = wm.sum()
    while True:
        j, p, q, g = _winners(m, mc, mr, wm)
        if not j.numel():
            break
        k = mr[m.row[p]]
        if select:
            order = torch.argsort(j, stable=True)
            order = order[torch.argsort(g[order], descending=True, stable=True)]
            rank = torch.empty_like(order)
            rank[order] = torch.arange(order.numel(), device=DEV)
            live = torch.ones_like(j, dtype=torch.bool)
            keep = torch.zeros_like(live)
            used = torch.zeros(n, device=DEV, dtype=torch.bool)
            while bool(live.any()):
                r, a, b = rank[live], j[live], k[live]
                first = _amin(n, torch.cat([a, b]), torch.cat([r, r]))
                now = live & (first[j] == rank) & (first[k] == rank)
                keep |= now
                used[j[now]] = True
                used[k[now]] = True
                live &= ~(used[j] | used[k])
        else:
            root = torch.zeros(n, device=DEV, dtype=torch.bool)
            root[j] = True
            ok = ~root[k]
            best = _amax(n, k[ok], g[ok])
            ok &= g == best[k]
            low = _amin(n, k[ok], j[ok])
            keep = ok & (low[k] == j)
        j, p, q, k = j[keep], p[keep], q[keep], k[keep]
        i, mj = m.row[p], mc[j]
        mc[j], mr[i], mc[k], mr[mj] = i, j, mj, k
        wm[j], wm[k] = m.w[p], m.w[q]
    return mc.int(), torch.stack([win, wm.sum()])


def _greedy(m):
    n = m.n
    order = torch.argsort(m.row * n + m.col)
    order = order[torch.argsort(m.w[order], descending=True, stable=True)]
    rank = torch.empty_like(order)
    rank[order] = torch.arange(order.numel(), device=DEV)
    mc, mr, wm = _full(n, -1), _full(n, -1), _full(n, 0.0, torch.float64)
    p = torch.arange(rank.numel(), device=DEV)
    while p.numel():
        r = rank[p]
        now = p[(r == _amin(n, m.col[p], r)[m.col[p]]) & (r == _amin(n, m.row[p], r)[m.row[p]])]
        mc[m.col[now]], mr[m.row[now]], wm[m.col[now]] = m.row[now], m.col[now], m.w[now]
        p = p[(mc[m.col[p]] < 0) & (mr[m.row[p]] < 0)]
    return mc, wm.sum().reshape(1)


def _mcm(m, mate):
    n = m.n
    mc = mate.to(DEV).long().clone()
    mr = _full(n, -1)
    have = torch.nonzero(mc >= 0).flatten()
    mr[mc[have]] = have
    while True:
        root, par, end = _full(n, -1), _full(n, -1), _full(n, -1)
        front = torch.nonzero(mc < 0).flatten()
        root[front] = front
        while front.numel():
            deg = m.ptr[front + 1] - m.ptr[front]
            c = torch.repeat_interleave(front, deg)
            p = torch.arange(c.numel(), device=DEV) + torch.repeat_interleave(
                m.ptr[front] - (torch.cumsum(deg, 0) - deg), deg)
            r = m.row[p]
            ok = (r != mc[c]) & (par[r] < 0)
            c, p, r = c[ok], p[ok], r[ok]
            top = _amax(n, r, m.w[p])
            s = m.w[p] == top[r]
            low = _amin(n, r[s], c[s])
            rows = torch.nonzero(low < BIG).flatten()
            par[rows] = low[rows]
            tree, c2 = root[low[rows]], mr[rows]
            fr = c2 < 0
            e, t = rows[fr], tree[fr]
            s = top[e] == _amax(n, t, top[e])[t]
            best = _amin(n, t[s], e[s])
            end = torch.where(best < BIG, best, end)
            root[c2[~fr]] = tree[~fr]
            front = c2[~fr]
            front = front[end[root[front]] < 0]
        r = end[(mc < 0) & (end >= 0)]
        if not r.numel():
            return mc
        while r.numel():
            c = par[r]
            old = mc[c]
            mc[c], mr[r] = r, c
            r = old[old >= 0]


def exact(case, seed):
    op = case["op"]
    st = prepare(case, seed)
    if op == "serve":
        got = [_phase(_M(n, *a[:3]), a[3], 0) for n, a, _ in st["reqs"]]
        return {"mates": [x[0].cpu() for x in got][:30], "counts": None,
                "weights": torch.stack([x[1] for x in got])}
    m = _M(st["n"], st["colptr"], st["rowidx"], st["weight"])
    if op == "mcm":
        return {"mate": _mcm(m, st["mate"]).int(), "counts": None}
    if op == "greedy":
        mc, w = _greedy(m)
        return {"mate": mc.int(), "counts": None, "weights": w}
    if op == "weights":
        a = m.w.abs()
        v = a / _amax(m.n, m.col, a)[m.col]
        x = v / _amax(m.n, m.row, v)[m.row]
        out = torch.zeros(_room(case), device=DEV, dtype=torch.float64)
        out[:x.numel()] = torch.log(x) if case["mode"] else x
        return {"weight": out}
    if op in ("search", "noalloc"):
        mc = st["mate"].long()
        ids = torch.arange(m.n, device=DEV)
        mr = torch.empty_like(mc)
        mr[mc] = ids
        j, p, _, g = _winners(m, mc, mr, m.w[torch.searchsorted(m.key, ids * m.n + mc)])
        gain, row = _full(m.n, 0.0, torch.float64), _full(m.n, -1)
        gain[j], row[j] = g, m.row[p]
        return {"gain": gain, "row": row.int(), "counts": None}
    mate = st.get("mate")
    if op == "pipeline":
        mate = _mcm(m, _greedy(m)[0])
    mc, w = _phase(m, mate, case.get("select", 0))
    return {"mate": mc, "counts": None, "weights": w}
