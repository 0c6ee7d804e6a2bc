"""The integer division and logarithm of the weights (csrc/awpm_fixed.h),
compiled for the CPU: quotients equal to the IEEE division bit for bit, and
refused exactly where an operand or the quotient is not normal; logarithms
within 0.53 units in the last place of the exact value."""
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1801_09809_gb300", "csrc")
TINY = np.finfo(np.float64).tiny


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_math")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC, "-o", exe,
                           os.path.join(HERE, "fixed_math.cpp")])

    def run(mode, x):
        out = subprocess.run([exe, mode], input=np.ascontiguousarray(x, np.float64).tobytes(),
                             stdout=subprocess.PIPE, check=True).stdout
        return np.frombuffer(out, np.float64)
    return run


def mantissas(rng, m):
    """Mantissas with the edges over-represented."""
    x = rng.integers(0, 1 << 52, m, dtype=np.int64)
    pick = rng.integers(0, 8, m)
    x = np.where(pick == 0, rng.integers(0, 4, m), x)
    x = np.where(pick == 1, (1 << 52) - 1 - rng.integers(0, 4, m), x)
    return x


def test_quotients(harness):
    rng = np.random.default_rng(1)
    m = 400_000
    ma, mb = mantissas(rng, m), mantissas(rng, m)
    mb = np.where(rng.integers(0, 5, m) == 0, np.clip(ma + rng.integers(-2, 3, m), 0, (1 << 52) - 1), mb)
    wide = rng.integers(0, 3, m) == 0
    ea = np.where(wide, rng.integers(0, 2047, m), rng.integers(1000, 1050, m))
    eb = np.where(wide, rng.integers(0, 2047, m), rng.integers(1000, 1050, m))
    a = ((ea << 52) | ma).view(np.float64)
    b = ((eb << 52) | mb).view(np.float64)
    keep = (a > 0) & (b > 0)
    a, b = a[keep], b[keep]
    got = harness("d", np.stack([a, b], 1))
    with np.errstate(over="ignore", under="ignore"):
        ref = a / b
    took = got != -1.0
    assert np.array_equal(got[took], ref[took])
    # refused: operands or quotients outside the normal numbers, and at most
    # the outermost binades inside them
    normal = (a >= TINY) & (b >= TINY) & (ref >= 2 * TINY) & (ref < 2.0 ** 1022)
    assert np.all(took[normal])
    assert not np.any(took[(a < TINY) | (b < TINY) | (ref < TINY)])


def test_logarithms(harness):
    rng = np.random.default_rng(2)
    m = 4000
    k = np.where(rng.integers(0, 2, m) == 0, rng.integers(0, 3, m), rng.integers(0, 1022, m))
    x = (((1022 - k) << 52) | mantissas(rng, m)).view(np.float64)
    edges = 0.5 + np.arange(513) / 1024.0                      # the table's interval ends
    near = 1.0 - 2.0 ** -np.arange(1, 54)                      # and the approach to 1
    x = np.concatenate([x, edges[:-1], np.nextafter(edges, 0), near, [TINY]])
    got = harness("l", x)
    getcontext().prec = 60
    worst = 0.0
    for v, g in zip(x.tolist(), got.tolist()):
        ref = Decimal(v).ln()
        ulp = float(np.spacing(abs(float(ref))))
        worst = max(worst, abs(float(Decimal(g) - ref)) / ulp)
    # half a unit from the final rounding; the rest from the truncated terms
    # (2^-58 of the result, 2^-5 of a unit)
    assert worst <= 0.5 + 2.0 ** -5
