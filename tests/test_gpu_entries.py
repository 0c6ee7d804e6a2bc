"""The entry pass at the edges of its 128-entry blocks and 4-entry lanes (needs
a GPU): sizes around the blocks' ends, columns starting and ending anywhere in
a lane, unaligned arrays, errors at every place of a block.  The search's
results depend on the signatures and filters that this pass builds."""
import numpy as np
import pytest

import oracle
from gpu_helpers import assert_same_as_oracle
from paper_1801_09809_gb300 import awpm, gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_09809_gb300 import build
    build.build()
    return _t


@pytest.fixture
def ctx(torch):
    # hash lookups build no Bloom filters, binary search does; the row-marking
    # lookup keeps these small problems on the general path
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_ROWMARK)
    yield c
    awpm.awpm_destroy(c)


def shaped(degrees, seed):
    """A matrix with the given column degrees and a planted matching."""
    rng = np.random.default_rng(seed)
    n = len(degrees)
    mate = rng.permutation(n).astype(np.int32)
    rows = []
    for j, d in enumerate(degrees):
        others = rng.permutation(n)[:d]
        r = np.unique(np.append(others, mate[j]))
        while r.size > d and r.size > 1:
            drop = rng.integers(0, r.size)
            if r[drop] != mate[j]:
                r = np.delete(r, drop)
        rows.append(r)
    colptr = np.zeros(n + 1, np.int32)
    np.cumsum([r.size for r in rows], out=colptr[1:])
    rowidx = np.concatenate(rows).astype(np.int32)
    w = rng.integers(-4, 5, rowidx.size).astype(np.float64)
    return gen.Graph(n, colptr, rowidx, w, mate, "shaped")


def on_device(torch, a, shift):
    """A copy on the GPU, `shift` elements past an aligned address."""
    buf = torch.zeros(a.size + shift, dtype=torch.from_numpy(a[:1]).dtype, device="cuda")
    buf[shift:].copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return buf[shift:]


CASES = {
    "ones": [1] * 300, "twos": [2] * 130, "threes": [3] * 129, "fours": [4] * 96,
    "long_between": [1, 140, 1, 2, 33, 3, 128, 5, 1, 1, 260, 4, 31, 32] + [1] * 300,
    "block": [4] * 32, "one_past": [4] * 32 + [1], "one_short": [4] * 31 + [3],
    "mixed": list(np.random.default_rng(5).integers(1, 9, 500)),
    "cut": [127, 2, 126, 1, 128, 129] + [1] * 200,
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("lookup", [awpm.LOOKUP_ROWMARK, awpm.LOOKUP_HASH])
def test_shapes(torch, name, shift, lookup):
    g = shaped(CASES[name], 9990)
    ref, rst, _ = oracle.get().improve(g)
    c = awpm.awpm_create(device=0, lookup=lookup)
    try:
        cp, ri, w = on_device(torch, g.colptr, 0), on_device(torch, g.rowidx, shift), \
            on_device(torch, g.weight, shift)
        m = torch.from_numpy(g.mate).cuda()
        out = torch.empty_like(m)
        st = awpm.awpm_improve_ctx(c, g.n, cp, ri, w, m, out)
        assert_same_as_oracle(g, out.cpu().numpy(), st, ref, rst, name)
    finally:
        awpm.awpm_destroy(c)


@pytest.mark.parametrize("shift", [0, 1])
def test_long_columns_with_filters(torch, shift):
    """Binary search with Bloom filters: hubs among short columns."""
    g = gen.rmat(20000, 12, 9991)
    ref, rst, _ = oracle.get().improve(g)
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH)
    try:
        ri, w = on_device(torch, g.rowidx, shift), on_device(torch, g.weight, shift)
        cp, m = on_device(torch, g.colptr, 0), torch.from_numpy(g.mate).cuda()
        out = torch.empty_like(m)
        st = awpm.awpm_improve_ctx(c, g.n, cp, ri, w, m, out)
        assert_same_as_oracle(g, out.cpu().numpy(), st, ref, rst, "rmat")
    finally:
        awpm.awpm_destroy(c)


def test_errors_anywhere(ctx, torch):
    g = shaped([5] * 80, 9992)
    cp, m = (torch.from_numpy(x).cuda() for x in (g.colptr, g.mate))
    out = torch.empty_like(m)

    def code(rowidx, weight):
        ri, w = torch.from_numpy(rowidx).cuda(), torch.from_numpy(weight).cuda()
        try:
            awpm.awpm_improve_ctx(ctx, g.n, cp, ri, w, m, out)
        except awpm.AwpmError as e:
            return e.name
        return "OK"

    for p in list(range(0, 12)) + list(range(120, 136)) + [g.nnz - 1]:
        w = g.weight.copy()
        w[p] = np.inf
        assert code(g.rowidx, w) == "NONFINITE", p
        r = g.rowidx.copy()
        r[p] = g.n
        assert code(r, g.weight) == "INVALID_ARG", p
        if p not in g.colptr:
            r = g.rowidx.copy()
            r[p] = r[p - 1]
            assert code(r, g.weight) == "UNSORTED_OR_DUP", p
    assert code(g.rowidx, g.weight) == "OK"


@pytest.mark.parametrize("mean", [39, 40])
def test_filters_of_ordinary_columns(torch, mean):
    """Columns of 31 to 66 rows (and one of 1,000) on both sides of the average from which columns
    of more than 32 rows have a Bloom filter, a search and a whole solve."""
    rng = np.random.default_rng(mean)
    d = rng.choice([31, 32, 33, 34, 45, 64, 65, 66], 1400, p=[.3, .2, .2, .1, .05, .05, .05, .05])
    d[:1300] += (mean * 1400 - d.sum()) // 1300
    d[-1] += mean * 1400 - d.sum()
    g = shaped(list(d), 9991)
    assert g.nnz == mean * g.n and g.nnz > 40960
    ref, rst, _ = oracle.get().improve(g)
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH)
    try:
        out = np.empty(g.n, np.int32)
        st = awpm.awpm_improve_ctx(c, g.n, g.colptr, g.rowidx, g.weight, g.mate, out)
        assert_same_as_oracle(g, out, st, ref, rst)
        gain, row = np.empty(g.n), np.empty(g.n, np.int32)
        awpm.awpm_search(c, g.n, g.colptr, g.rowidx, g.weight, g.mate, gain, row)
        want_gain, want_row, _ = oracle.get().step_c(g)
        assert np.array_equal(gain, want_gain) and np.array_equal(row, want_row)
    finally:
        awpm.awpm_destroy(c)
