"""Weights from matrix values at the edges of the entry-parallel kernels
(needs a GPU): empty columns, columns longer than a tile, sizes around tile
ends, values and quotients outside the normal numbers."""
import numpy as np
import pytest

from paper_1801_09809_gb300 import awpm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_09809_gb300 import build
    build.build()
    c = awpm.awpm_create(device=0)
    yield c
    awpm.awpm_destroy(c)


def matrix(degrees, seed, span):
    """Random rows, `degrees[j]` per column; values 10^U(-span, min(span, 308))."""
    rng = np.random.default_rng(seed)
    n = len(degrees)
    colptr = np.zeros(n + 1, np.int32)
    np.cumsum(degrees, out=colptr[1:])
    rows = [np.sort(rng.choice(n, d, replace=False)) for d in degrees]
    rowidx = np.concatenate(rows).astype(np.int32) if rows else np.zeros(0, np.int32)
    a = 10.0 ** rng.uniform(-span, min(span, 308), rowidx.size) * rng.choice([-1.0, 1.0], rowidx.size)
    a[a == 0.0] = 5e-324
    return n, colptr, rowidx, a


def reference(n, colptr, rowidx, a, mode):
    col = np.repeat(np.arange(n), np.diff(colptr))
    with np.errstate(all="ignore"):
        cm = np.zeros(n)
        np.maximum.at(cm, col, np.abs(a))
        v = np.abs(a) / cm[col]
        rm = np.zeros(n)
        np.maximum.at(rm, rowidx, v)
        x = v / rm[rowidx]
        return np.log(x) if mode else x


# sizes at the ends of the ranges of the three forms (tiles of 32 entries, and
# with nnz / 6 columns a sixth of their number for the columns in the first)
SIZES = [384 * 32 + x for x in (-1, 0, 1, 32)] + [10559 + x for x in (-31, 0, 1)]
SIZES += [4096 * 32 + x for x in (-31, 0, 1)]

CASES = {
    "empty_columns": [0, 0, 3, 0, 31, 32, 33, 0, 1, 0, 0, 64, 65, 0, 0, 1] + [0, 1, 2] * 40,
    "hub": [200] + [1] * 199,
    "one_tile": [4] * 8,
    "one_past": [4] * 8 + [1],
    "one": [1],
    "all_but_one_empty": [0] * 50 + [37] + [0] * 49,
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("span", [2, 300, 323])
@pytest.mark.parametrize("mode", [0, 1])
def test_edges(ctx, name, span, mode):
    import torch
    n, colptr, rowidx, a = matrix(CASES[name], 7 + span, span)
    want = reference(n, colptr, rowidx, a, mode)
    for in_place in (False, True):
        cp, ri, av = (torch.from_numpy(x).cuda() for x in (colptr, rowidx, a))
        out = av if in_place else torch.empty_like(av)
        awpm.awpm_weights(ctx, n, cp, ri, av, mode, out)
        got = out.cpu().numpy()
        if mode == 0:
            assert np.array_equal(got, want, equal_nan=True)
        else:
            # numpy's logarithm is within an ulp of the exact value, the
            # library's within one too
            fine = np.isfinite(want)
            assert np.array_equal(got[~fine], want[~fine], equal_nan=True)
            assert np.all(np.abs(got[fine] - want[fine]) <= 2 * np.spacing(np.abs(want[fine])))


@pytest.mark.parametrize("nnz", SIZES)
def test_forms(ctx, nnz):
    """Either side of the lines between the forms, with a long column, empty
    ones and a remainder: the quotients bit for bit, in place too."""
    import torch
    rng = np.random.default_rng(nnz)
    n = nnz // 6
    degrees = rng.integers(0, 10, n)
    degrees[n // 3] = 1500
    while degrees.sum() != nnz:
        j = rng.integers(0, n)
        if degrees.sum() < nnz:
            degrees[j] += 1
        elif degrees[j]:
            degrees[j] -= min(degrees[j], degrees.sum() - nnz)
    n, colptr, rowidx, a = matrix(list(degrees), nnz, 300)
    want = reference(n, colptr, rowidx, a, 0)
    for in_place in (False, True):
        cp, ri, av = (torch.from_numpy(x).cuda() for x in (colptr, rowidx, a))
        out = av if in_place else torch.empty_like(av)
        awpm.awpm_weights(ctx, n, cp, ri, av, 0, out)
        assert np.array_equal(out.cpu().numpy(), want, equal_nan=True)
    # what is refused: a value of zero, a row out of range, a bad column pointer
    for k in range(3):
        c2, r2, a2 = colptr.copy(), rowidx.copy(), a.copy()
        if k == 0:
            a2[nnz - 1] = 0.0
        elif k == 1:
            r2[nnz // 2] = n
        else:
            c2[n // 2] = nnz + 1
        cp, ri, av = (torch.from_numpy(x).cuda() for x in (c2, r2, a2))
        with pytest.raises(awpm.AwpmError):
            awpm.awpm_weights(ctx, n, cp, ri, av, 0, torch.empty_like(av))


@pytest.mark.parametrize("n", [368 * 32 + 31, 369 * 32, 4096 * 32 + 31, 4097 * 32])
def test_mostly_empty(ctx, n):
    """500 entries (16 tiles) in so many columns that n decides the form."""
    import torch
    rng = np.random.default_rng(n)
    key = np.unique(rng.integers(0, n * n, 500))
    assert key.size == 500
    colptr = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int32)
    rowidx, a = (key % n).astype(np.int32), rng.standard_normal(500)
    want = reference(n, colptr, rowidx, a, 0)
    cp, ri, av = (torch.from_numpy(x).cuda() for x in (colptr, rowidx, a))
    out = torch.empty_like(av)
    awpm.awpm_weights(ctx, n, cp, ri, av, 0, out)
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("where", ["device", "in_place", "host"])
def test_budget_without_room(ctx, mode, where):
    """A budget that holds the row maxima and the staged arrays but neither the
    columns' scales nor the tiles' columns gives the same bits."""
    import torch
    # (more tiles than the small matrices', which take the thin form anyway)
    n, colptr, rowidx, a = matrix(CASES["empty_columns"] * 450 + [3000] + [0, 1, 2, 40] * 100, 5,
                                  300)
    assert a.size > 4096 * 32

    def solve(c, a):
        if where == "host":
            out = np.empty_like(a)
            awpm.awpm_weights(c, n, colptr, rowidx, a, mode, out)
            return out
        cp, ri, av = (torch.from_numpy(x).cuda() for x in (colptr, rowidx, a))
        out = av if where == "in_place" else torch.empty_like(av)
        awpm.awpm_weights(c, n, cp, ri, av, mode, out)
        return out.cpu().numpy()

    full = awpm.awpm_create(device=0)
    want = solve(full, a)
    held = awpm.awpm_memory_held(full)[0]
    awpm.awpm_destroy(full)
    # Allocations take an eighth of headroom while it fits, so a budget short of
    # what the full form held by 18 n (its scales, with their headroom) has
    # room for the thin form; the full form could save only the headroom of its
    # last allocation, at most nnz bytes.
    assert a.size < 18 * n
    budget = held - 18 * n
    c = awpm.awpm_create(device=0, mem_budget_bytes=budget)
    try:
        assert np.array_equal(solve(c, a), want, equal_nan=True)
        assert awpm.awpm_memory_held(c)[1] <= budget
        bad = a.copy()
        bad[a.size // 2] = 0.0
        with pytest.raises(awpm.AwpmError):
            solve(c, bad)
        assert np.array_equal(solve(c, a), want, equal_nan=True)
    finally:
        awpm.awpm_destroy(c)
