"""Greedy and maximum matching around the sizes where their loops move from one
cluster to the graph (needs a GPU), empty columns and unmatched columns
included: equal to the oracle on both sides of the line; and the end of a
maximum matching whose bounded retries give up."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import oracle
from paper_1801_09809_gb300 import awpm, gen

pytestmark = pytest.mark.gpu
# most entries of a problem of nnz / 6 columns in one cluster (the maximum
# matching counts 32 columns as a tile of 32 entries)
GREEDY, MCM = 3584 * 32, 182591


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


def sized(nnz, seed, integer_weights):
    """About n = nnz / 6 columns, exactly nnz entries: a random graph with
    entries added to its last columns."""
    rng = np.random.default_rng(seed)
    n = nnz // 6
    g = gen.random_sparse(n, 5, seed)
    have = g.nnz
    deg = np.diff(g.colptr)
    add = np.zeros(n, np.int64)
    add[n - (nnz - have):] = 1
    rows = [g.rowidx[g.colptr[j]:g.colptr[j + 1]] for j in range(n)]
    for j in np.nonzero(add)[0]:
        r = int(rng.integers(0, n))
        while r in rows[j]:
            r = (r + 1) % n
        rows[j] = np.sort(np.append(rows[j], r)).astype(np.int32)
    colptr = np.zeros(n + 1, np.int32)
    np.cumsum(deg + add, out=colptr[1:])
    rowidx = np.concatenate(rows).astype(np.int32)
    assert rowidx.size == nnz
    w = rng.integers(-3, 4, nnz).astype(np.float64) if integer_weights else rng.standard_normal(nnz)
    return gen.Graph(n, colptr, rowidx, w, g.mate, f"sized({nnz})")


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("nnz", [GREEDY - 31, GREEDY, GREEDY + 1])
def test_greedy(ctx, nnz, ties):
    g = sized(nnz, 9970, ties)
    ref, rst = oracle.get().greedy(g)
    out = np.empty(g.n, np.int32)
    st = awpm.awpm_greedy(ctx, g.n, g.colptr, g.rowidx, g.weight, out)
    assert np.array_equal(out, ref)
    assert st["cardinality"] == rst["cardinality"] and st["rounds"] == rst["rounds"]


def emptied(nnz, seed):
    """As sized(), with three columns empty."""
    g = sized(nnz + 120, seed, True)
    cp, col = g.colptr, np.repeat(np.arange(g.n), np.diff(g.colptr))
    keep = np.ones(g.nnz, bool)
    for j in (0, 5, g.n - 1):
        keep[cp[j]:cp[j + 1]] = False
    spare = np.nonzero(keep & (g.rowidx != g.mate[col]))[0]  # (the matched entries stay)
    keep[np.random.default_rng(4).choice(spare, keep.sum() - nnz, replace=False)] = False
    deg = np.bincount(col[keep], minlength=g.n)
    colptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    return gen.Graph(g.n, colptr, g.rowidx[keep], g.weight[keep], g.mate, f"emptied({nnz})")


@pytest.mark.parametrize("empty", [False, True])
@pytest.mark.parametrize("nnz,clusters", [(MCM - 31, True), (MCM, True), (MCM + 1, False)])
def test_mcm(ctx, nnz, clusters, empty):
    # (emptied() has 20 columns more for its entries)
    g = emptied(nnz - (40 if clusters else 20), 9980) if empty else sized(nnz, 9980, True)
    assert (-(-g.nnz // 32) + g.n // 32 <= 6656) == clusters
    rng = np.random.default_rng(3)
    mate = np.where(rng.random(g.n) < 0.1, -1, g.mate).astype(np.int32)
    if empty:
        mate[[0, 5, g.n - 1]] = -1
    ref, rst = oracle.get().mcm(g, mate)
    got = mate.copy()
    st = awpm.awpm_mcm(ctx, g.n, g.colptr, g.rowidx, g.weight, got)
    assert np.array_equal(got, ref)
    assert st["cardinality"] == int((ref >= 0).sum()) and st["phases"] == rst["phases"]


@pytest.mark.parametrize("n,on", [(60000, "0"), (70000, "0"), (200000, "1"), (230000, "1")])
def test_mcm_mostly_empty(monkeypatch, ctx, n, on):
    """4,000 entries: n decides whether the graph's first level is one cluster's
    (up to 65,567 columns), and between cluster and graph."""
    monkeypatch.setenv("AWPM_CLUSTER", on)
    rng = np.random.default_rng(n)
    key = np.unique(rng.integers(0, n // 50, 4000) * 50 * n + rng.integers(0, 1500, 4000))
    colptr = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int32)
    g = gen.Graph(n, colptr, (key % n).astype(np.int32),
                  rng.integers(0, 4, key.size).astype(np.float64), None, "mostly empty")
    start = np.full(n, -1, np.int32)
    ref, rst = oracle.get().mcm(g, start)
    got = start.copy()
    c = awpm.awpm_create(device=0)
    try:
        st = awpm.awpm_mcm(c, n, g.colptr, g.rowidx, g.weight, got)
    finally:
        awpm.awpm_destroy(c)
    assert np.array_equal(got, ref) and st["phases"] == rst["phases"]


@pytest.mark.parametrize("name", ["from_empty_and_from_greedy", "hand_tie_breaks", "bad_start",
                                  "hand_cases_equal_weights", "small_and_ties", "structures",
                                  "long_columns_and_equal_weights"])
def test_graph_form(monkeypatch, name):
    """The small problems of the maximum and the greedy matching's own tests, which
    take the cluster by their size, through the graph's loops."""
    import torch
    import test_gpu_greedy
    import test_gpu_mcm
    monkeypatch.setenv("AWPM_CLUSTER", "0")
    c = awpm.awpm_create(device=0)
    try:
        module = test_gpu_mcm if hasattr(test_gpu_mcm, "test_" + name) else test_gpu_greedy
        getattr(module, "test_" + name)(c, torch)
    finally:
        awpm.awpm_destroy(c)


NO_RETRIES = textwrap.dedent("""
    import sys
    sys.path[:0] = [{root!r}, {tests!r}]
    import numpy as np
    import pytest
    from paper_1801_09809_gb300 import awpm
    from test_gpu_clusters import MCM, sized
    assert awpm.LIB_PATH == {lib!r}
    ctx = awpm.awpm_create(device=0)
    for nnz in (2000, MCM, MCM + 32, 2 * MCM):
        g = sized(nnz, 9990, True)
        with pytest.raises(awpm.AwpmError) as e:
            awpm.awpm_mcm(ctx, g.n, g.colptr, g.rowidx, g.weight, np.full(g.n, -1, np.int32))
        assert e.value.name == "TIMEOUT", e.value.name
    awpm.awpm_destroy(ctx)
    print("NO_RETRIES_OK")
""")


def test_mcm_retries_given_up(ctx, tmp_path):
    """With no retries allowed (AWPM_CAS_RETRY_CAP = 0 in this file's kernels) a
    level's first offers raise the timeout bit while other blocks are still on
    their way into the level: the cluster and the graph form both end with
    AWPM_ERR_TIMEOUT."""
    from paper_1801_09809_gb300 import build
    obj, lib = str(tmp_path / "awpm_mcm.o"), str(tmp_path / "libawpm_retry.so")
    subprocess.check_call([build.NVCC, *build.ARCH, *build.FLAGS, "-DAWPM_CAS_RETRY_CAP=0", "-c",
                           os.path.join(build.CSRC, "awpm_mcm.cu"), "-o", obj])
    objs = [os.path.join(build.OBJDIR, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    subprocess.check_call([build.NVCC, "-shared", *build.ARCH, "-o", lib, obj,
                           *(o for o in objs if not o.endswith("awpm_mcm.o"))])
    tests = os.path.dirname(os.path.abspath(__file__))
    child = NO_RETRIES.format(root=build.ROOT, tests=tests, lib=lib)
    r = subprocess.run([sys.executable, "-c", child], env=dict(os.environ, AWPM_LIBRARY=lib),
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "NO_RETRIES_OK" in r.stdout, r.stdout + r.stderr
