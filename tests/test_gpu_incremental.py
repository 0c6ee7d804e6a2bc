"""The incremental passes (needs a GPU): forced on at every size (AWPM_INC=1, in
a child process, since the library reads it once) the existing parity and
record tests still hold, and so do cases of the small, the large and the
folded bitmap of changed rows and a budget without room for the buffer; by
rule, a problem of more than 3.1 M entries."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from gpu_helpers import assert_same_as_oracle, run_gpu
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


FORCED = os.environ.get("AWPM_INC") == "1"
forced = pytest.mark.skipif(not FORCED, reason="run by test_forced_on")


@pytest.mark.skipif(FORCED, reason="the child process")
@pytest.mark.parametrize("which", ["parity", "records", "incremental"])
def test_forced_on(torch, which):
    env = dict(os.environ, AWPM_INC="1")
    r = subprocess.run([sys.executable, "-m", "pytest", f"tests/test_gpu_{which}.py", "-q", "-x",
                        "-m", "gpu", "-p", "no:cacheprovider"], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]


CASES = {
    # n just past the small bitmap, many flips (large bitmap, exact)
    "banded_131073": lambda: gen.banded(131073, 5, 9801),
    # n past the large bitmap: folded, with false positives
    "banded_1200001": lambda: gen.banded(1200001, 3, 9802),
    # n below 2^17, many passes, equal gains
    "grid27_40": lambda: gen.stencil_3d(40, 9803),
    # hub columns and rows
    "rmat_100000": lambda: gen.rmat(100000, 12, 9804),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("opts", [{}, {"lookup": awpm.LOOKUP_HASH}, {"lookup": awpm.LOOKUP_ROWMARK},
                                  {"select": awpm.SELECT_GREEDY}, {"flags": awpm.FLAG_TIME_SEARCH},
                                  {"max_iters": 3}],
                         ids=["auto", "hash", "rowmark", "greedy", "timed", "three"])
def test_sizes(torch, name, opts):
    if not FORCED and name != "banded_1200001":
        pytest.skip("too small for the rule; run by test_forced_on")
    g = CASES[name]()
    if name == "grid27_40":
        # integer weights: many equal gains
        g.weight = np.round(g.weight * 4)
    ref, rst, _ = oracle.get().improve(g, select=opts.get("select", 0),
                                       max_iters=opts.get("max_iters", 0))
    c = awpm.awpm_create(device=0, **opts)
    try:
        for _ in range(2):  # the second solve starts from the first one's records
            got, st = run_gpu(c, g, torch=torch)
            assert_same_as_oracle(g, got, st, ref, rst, name)
    finally:
        awpm.awpm_destroy(c)


@forced
def test_budget_without_room(torch):
    """A budget that had room for a solve before the incremental buffer still
    has it: every pass then searches all, with the same result."""
    g = CASES["banded_131073"]()
    ref, rst, _ = oracle.get().improve(g)
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH)
    run_gpu(c, g, torch=torch)
    held, _ = awpm.awpm_memory_held(c)
    awpm.awpm_destroy(c)
    tiles = (g.nnz + 31) // 32
    buffer = 8 * tiles + 4 * g.n  # entry bits and old rows, without the bitmaps
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH, mem_budget_bytes=held - buffer)
    try:
        got, st = run_gpu(c, g, torch=torch)
        assert_same_as_oracle(g, got, st, ref, rst, "budget")
        assert awpm.awpm_memory_held(c)[1] <= held - buffer
    finally:
        awpm.awpm_destroy(c)


@forced
def test_budget_buffer_before_staging(torch):
    """Host arrays are staged after the incremental buffer is taken: where the
    two don't fit together the buffer is given back; and a buffer kept from an
    earlier solve makes room for another entry point."""
    g = CASES["banded_131073"]()
    ref, rst, _ = oracle.get().improve(g)
    sizes = []
    for passes in (0, 1):  # (one pass needs no buffer)
        c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH, max_iters=passes)
        run_gpu(c, g)
        sizes.append(awpm.awpm_memory_held(c)[0])
        awpm.awpm_destroy(c)
    held, buffer = sizes[0], sizes[0] - sizes[1]
    # The mate array is staged last, 4 n with n / 2 of headroom: a budget short
    # of all that by 2 n has no room for it beside the buffer.
    assert buffer > 2 * g.n
    budget = held - 2 * g.n
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH, mem_budget_bytes=budget)
    try:
        for _ in range(2):
            got, st = run_gpu(c, g)
            assert_same_as_oracle(g, got, st, ref, rst, "budget")
            assert awpm.awpm_memory_held(c)[1] <= budget
    finally:
        awpm.awpm_destroy(c)
    # the search's staged results (12 n, 13.5 n with headroom) have room only in
    # the buffer's place
    budget = held + max(0, 14 * g.n - buffer)
    assert budget < held + 12 * g.n
    c = awpm.awpm_create(device=0, lookup=awpm.LOOKUP_BSEARCH, mem_budget_bytes=budget)
    gain, row = np.empty(g.n), np.empty(g.n, np.int32)
    try:
        run_gpu(c, g)
        awpm.awpm_search(c, g.n, g.colptr, g.rowidx, g.weight, g.mate, gain, row)
        assert awpm.awpm_memory_held(c)[1] <= budget
        got, st = run_gpu(c, g)
        assert_same_as_oracle(g, got, st, ref, rst, "after the search")
    finally:
        awpm.awpm_destroy(c)
