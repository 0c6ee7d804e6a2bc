"""Solves of small matrices by a block (batches) or a cluster (single ones)
each (needs a GPU): the edges of the size classes against the oracle, both
sides of the line up to which a batch takes a block per matrix, inputs that go
back to the general path, and the existing parity, batch and record tests with
the small-matrix kernel switched off (in a child process), so that the general
path keeps its coverage at small sizes."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from gpu_helpers import assert_same_as_oracle, run_gpu, to_device
from paper_1801_09809_gb300 import awpm, gen

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_09809_gb300 import build
    build.build()
    return _t


@pytest.fixture(autouse=True)
def blocks(monkeypatch):
    """Batches go to the small-matrix kernel whenever their matrices fit it,
    whether that pays or not (read when a context is made)."""
    monkeypatch.setenv("AWPM_SMALL", "1")


@pytest.fixture
def ctx(torch):
    c = awpm.awpm_create(device=0)
    yield c
    awpm.awpm_destroy(c)


@pytest.mark.parametrize("which", ["parity", "batch", "records", "serve"])
def test_switched_off(torch, which):
    env = dict(os.environ, AWPM_SMALL="0")
    r = subprocess.run([sys.executable, "-m", "pytest", f"tests/test_gpu_{which}.py", "-q", "-x",
                        "-m", "gpu", "-p", "no:cacheprovider"], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]


def batch_check(ctx, torch, graphs, max_iters=0, host=False, times=2):
    """Solves a batch several times (each starts from the records that the one
    before left); returns the lookups used."""
    n_off, u = gen.union(graphs)
    if host:
        (cp, ri, w, m), off = (u.colptr, u.rowidx, u.weight, u.mate), n_off
        out = np.empty_like(m)
    else:
        cp, ri, w, m = to_device(u, torch)
        off = torch.from_numpy(n_off).cuda()
        out = torch.empty_like(m)
    used = []
    for _ in range(times):
        tot, per = awpm.awpm_improve_batch(ctx, len(graphs), off, cp, ri, w, m, out)
        used.append(tot["lookup_used"])
        got = gen.split(n_off, out if host else out.cpu().numpy())
        sums = dict.fromkeys(("candidates", "closing_found", "positive", "cycles_applied"), 0)
        for b, g in enumerate(graphs):
            ref, rst, _ = oracle.get().improve(g, max_iters=max_iters)
            assert np.array_equal(got[b], ref), (b, g.name)
            for k in ("iterations", "converged", "cycles_applied", "edge_checks"):
                assert per[b][k] == rst[k], (b, g.name, k)
            for k in sums:
                sums[k] += rst[k]
        assert {k: tot[k] for k in sums} == sums
    return used


def line_batches():
    """A batch on either side of the line (14,000 + 100 or 58 per tile of the
    slowest matrix against the union's 44,000 + 0.42 per tile): four alike, and
    one larger among many small ones."""
    small = [gen.banded(300, 9, 9970 + k) for k in range(100)]
    return [([gen.banded(1950, 5, 9971 + k) for k in range(4)], True),
            ([gen.banded(1965, 5, 9972 + k) for k in range(4)], False),
            (small + [gen.banded(3300, 5, 9973)], True),
            (small + [gen.banded(3800, 5, 9974)], False)]


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("which", range(4))
def test_lines(torch, monkeypatch, which, host):
    """Both sides of the line equal the oracle and go where they should: the
    third solve that a new context does as a union tries the hash lookup, the
    small-matrix kernel has none."""
    monkeypatch.delenv("AWPM_SMALL")
    graphs, blocks = line_batches()[which]
    c = awpm.awpm_create(device=0)
    try:
        used = batch_check(c, torch, graphs, host=host, times=3)
        assert used[2] == (awpm.LOOKUP_BSEARCH if blocks else awpm.LOOKUP_HASH)
    finally:
        awpm.awpm_destroy(c)


def test_class_edges(ctx, torch):
    """Matrices at the largest n of each class, one past it, tiny ones, long
    columns, an n without signatures, and more entries than the tile bitmap
    has room for."""
    graphs = [gen.banded(n, 5, 9900 + k) for k, n in
              enumerate((1, 2, 31, 32, 33, 2047, 2048, 2049, 7167, 7168, 7169, 14000, 20095, 20096))]
    graphs += [gen.random_small(600, 0.6, 9920, integer_weights=True), gen.stencil_3d(9, 9921),
               gen.rmat(3000, 20, 9922), gen.random_small(40, 0.9, 9923, integer_weights=True)]
    batch_check(ctx, torch, graphs)


def test_one_past_the_largest(ctx, torch):
    batch_check(ctx, torch, [gen.banded(20097, 3, 9930), gen.banded(50, 3, 9931)])


def test_pass_cap(torch):
    c = awpm.awpm_create(device=0, max_iters=2)
    try:
        batch_check(c, torch, [gen.banded(500 + 700 * k, 9, 9940 + k) for k in range(4)], 2)
    finally:
        awpm.awpm_destroy(c)


def test_budget_for_blocks_only(torch, monkeypatch):
    """A batch that the rule makes a union, under a budget with room for the blocks
    only, is solved by them, within the budget."""
    graphs = [gen.banded(7000 + k, 9, 9980 + k) for k in range(4)]

    def context(small, budget):
        monkeypatch.setenv("AWPM_SMALL", small)
        return awpm.awpm_create(device=0, mem_budget_bytes=budget)

    c = context("1", 0)
    batch_check(c, torch, graphs)
    budget = awpm.awpm_memory_held(c)[1]
    awpm.awpm_destroy(c)
    c = context("0", budget)
    with pytest.raises(awpm.AwpmError) as e:
        batch_check(c, torch, graphs)
    assert e.value.name == "BUDGET"
    awpm.awpm_destroy(c)
    c = context("", budget)
    try:
        used = batch_check(c, torch, graphs, times=4)
        assert used == [awpm.LOOKUP_BSEARCH] * 4
        assert awpm.awpm_memory_held(c)[1] <= budget
    finally:
        awpm.awpm_destroy(c)


@pytest.mark.parametrize("make", [
    lambda: gen.random_small(1, 1.0, 1), lambda: gen.random_small(33, 0.5, 2, integer_weights=True),
    lambda: gen.banded(2048, 15, 3), lambda: gen.banded(2049, 15, 4), lambda: gen.stencil_2d(90, 5),
    # past the entries' limit: found by the kernel (n small) or before it
    lambda: gen.random_small(400, 0.9, 6, integer_weights=True), lambda: gen.banded(4600, 9, 7),
    lambda: gen.rmat(2000, 30, 8)],
    ids=["one", "tiny", "n2048", "n2049", "grid5", "dense400", "nnz41k", "rmat2000"])
def test_single(ctx, torch, make):
    g = make()
    ref, rst, _ = oracle.get().improve(g)
    for host in (False, True, False):
        got, st = run_gpu(ctx, g, torch=torch, host=host)
        assert_same_as_oracle(g, got, st, ref, rst, g.name)


@pytest.mark.parametrize("batch", [False, True])
def test_errors_named_in_place(ctx, torch, batch):
    """Broken inputs get the general path's error class, also with mate_out the
    same array as mate_in; the context solves correctly afterwards."""
    g = gen.banded(300, 5, 9950)
    others = [gen.banded(100, 3, 9951), gen.banded(900, 7, 9952)] if batch else []

    def call(h):
        graphs = others[:1] + [h] + others[1:]
        n_off, u = gen.union(graphs)
        cp, ri, w, m = to_device(u, torch)
        if batch:
            awpm.awpm_improve_batch(ctx, len(graphs), n_off, cp, ri, w, m, m)
        else:
            awpm.awpm_improve_ctx(ctx, u.n, cp, ri, w, m, m)
        return gen.split(n_off, m.cpu().numpy())

    def broken(f):
        h = g.copy()
        f(h)
        return h

    def swap_rows(h):
        h.rowidx[[4, 5]] = h.rowidx[[5, 4]]

    def bad_weight(h):
        h.weight[7] = np.nan

    def same_mate(h):
        h.mate[3] = h.mate[2]

    def both(h):
        swap_rows(h)
        same_mate(h)

    for f, name in ((swap_rows, "UNSORTED_OR_DUP"), (bad_weight, "NONFINITE"),
                    (same_mate, "NOT_PERFECT"), (both, "UNSORTED_OR_DUP")):
        with pytest.raises(awpm.AwpmError) as e:
            call(broken(f))
        assert e.value.name == name
    ref, _, _ = oracle.get().improve(g)
    assert np.array_equal(call(g)[1 if batch else 0], ref)


@pytest.mark.parametrize("off", [-1, 1])
@pytest.mark.parametrize("n", [300, 3000])
def test_stated_entries(ctx, torch, n, off):
    """A served request whose stated number of entries is not colptr[n] is
    refused, by one too many as by one too few (the arrays are one longer than
    the matrix), and the same request with the right number is solved."""
    g = gen.banded(n, 5, 9960)
    cp, ri, w, m = to_device(g, torch)
    ri, w = torch.cat([ri, ri[:1]]), torch.cat([w, w[:1]])
    out = torch.empty_like(m)
    with pytest.raises(awpm.AwpmError) as e:
        awpm.awpm_wait(ctx, awpm.awpm_submit(ctx, n, cp, ri, w, m, out, nnz=g.nnz + off))
    assert e.value.name == "INVALID_ARG"
    awpm.awpm_wait(ctx, awpm.awpm_submit(ctx, n, cp, ri, w, m, out, nnz=g.nnz))
    assert np.array_equal(out.cpu().numpy(), oracle.get().improve(g)[0])
