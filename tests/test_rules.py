"""The index arithmetic and size rules of the library (csrc/awpm_rules.h),
compiled for the CPU."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1801_09809_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("rules") / "rules")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + CSRC, "-o", exe,
                           os.path.join(HERE, "rules.cpp")])

    def call(*args):
        out = subprocess.run([exe, *map(str, args)], stdout=subprocess.PIPE, check=True).stdout
        return int(out.split()[0])
    return call


def test_tiles_past_the_last_never_wrap(rule):
    """The search looks ahead by up to three rounds of two tiles per warp: with
    the most entries accepted those tiles' lanes are still past the end, while
    t * 32 + lane would be negative in 32 bits, hence "below nnz"."""
    nnz = rule("max_entries")
    ntiles = -(-nnz // 32)
    ahead = 4 * 2 * 160 * 32  # rounds x tiles x SMs x warps, rounded up
    wrapped = ((ntiles + ahead) * 32 + 2 ** 31) % 2 ** 32 - 2 ** 31
    assert wrapped < 0
    for t in (ntiles, ntiles + 1, ntiles + 2, ntiles + ahead):
        for lane in (0, 31):
            assert nnz <= rule("tile_pos", t, ntiles, lane) < 2 ** 31
    for t in (0, 1, ntiles - 1):
        for lane in (0, 31):
            assert rule("tile_pos", t, ntiles, lane) == t * 32 + lane


def test_batches_by_work(rule):
    """A block per matrix where the largest matrix is no more than its share of
    the work: not for few large matrices, nor dense ones, whatever their n."""
    def blocks(*matrices):
        return rule("blocks_pay", *(x for n, tiles, count in matrices for x in (n, tiles) * count))
    assert blocks((300, 84, 1)) and blocks((300, 84, 4)) and blocks((300, 84, 1024))
    assert not blocks((2000, 562, 1)) and not blocks((2000, 562, 16)) and blocks((2000, 562, 256))
    assert not blocks((20000, 5624, 1)) and not blocks((20000, 5624, 64))
    assert blocks((20000, 5624, 256))
    assert not blocks((1000, 15750, 4)) and not blocks((10000, 152700, 4))
    assert not blocks((600, 167, 512), (20000, 10620, 1))
    # the line for four matrices of the smallest class
    assert blocks((1950, 305, 4)) and not blocks((1960, 306, 4))
    # empty matrices, and one class's largest n beside the next
    assert blocks((0, 0, 3)) and blocks((0, 0, 100), (20, 3, 1))
    assert not blocks((2048, 400, 4)) and blocks((2049, 400, 4)) and blocks((7169, 800, 4))


def test_mostly_empty_matrices(rule):
    """Columns count as well as entries where a form walks all of them: few
    entries in millions of columns do not go to eight blocks."""
    most = 2 ** 31 - 1
    assert rule("mcm_cluster", 6000, 20000) and not rule("mcm_cluster", 6000, 32000)
    assert rule("mcm_cluster", 32, 131072) and not rule("mcm_cluster", 32, 262144)
    assert not rule("mcm_cluster", 1, most) and not rule("mcm_cluster", 67108862, most)
    assert [rule("weights_form", 16, n) for n in (100, 11807, 11808, 131103, 131104, most)] == \
        [0, 0, 1, 1, 2, 2]
    assert [rule("weights_form", t, 1000) for t in (353, 354, 4096, 4097)] == [0, 1, 1, 2]


def test_small_solve_with_too_many_entries(rule):
    """A solve of at most 40,960 entries that comes back undone was refused for
    something else: its size class goes on without the number read first."""
    assert [rule("small_too_many", z) for z in (0, 300, 40960, 40961, 2 ** 31 - 1)] == [0, 0, 0, 1, 1]
