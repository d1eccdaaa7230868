"""The block fixed-point arithmetic of the FP64 kernels (csrc/fx.cuh), compiled on
the CPU from its own source: values survive the round trip through a block to the
block's last place, sums of products are exact to two units, and what is not a
normal number is treated as documented."""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def dump(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fx") / "fx_dump")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + os.path.join(CUDA, "include"),
                    "-I" + os.path.join(ROOT, "paper_2510_00998_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fx_dump.cpp"), "-o", exe], check=True)

    def run(a, x):
        n, k = x.shape
        text = f"{n} {k}\n" + "\n".join(" ".join(f"{float(p).hex()} {float(q).hex()}" for p, q in zip(ra, rx))
                                        for ra, rx in zip(a, x))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        rows = [[float.fromhex(v) if "n" not in v else float(v) for v in line.split()] for line in out.splitlines()]
        return np.array(rows)
    return run


@pytest.mark.parametrize("spread", [0, 12, 40, 200])
@pytest.mark.parametrize("k", [2, 4, 7])
def test_blocks_keep_59_bits_and_sums_two_units(dump, spread, k):
    rng = np.random.default_rng(7 * k + spread)
    x = rng.normal(size=(40, k)) * 2.0 ** rng.integers(-spread, spread + 1, size=(40, k)) * 2.0 ** rng.integers(-300, 300)
    a = rng.uniform(-1, 1, size=(40, k))
    out = dump(a, x)
    for ra, rx, ro in zip(a, x, out):
        unit = Fraction(2) ** (int(np.frexp(np.abs(rx).max())[1]) - 1 - 59)
        for v, w in zip(rx, ro):
            # cut to the block's unit, then rounded to 53 bits
            assert abs(Fraction(float(w)) - Fraction(float(v))) <= unit + abs(Fraction(float(v))) / 2 ** 53
        # a is cut to 2^-59 (times |x| < 2^60 units), x to a unit, the low product dropped:
        # k units each at most, 2^5 of which make a unit of the sum's value
        exact = sum(Fraction(float(p)) * Fraction(float(q)) for p, q in zip(ra, rx))
        assert abs(Fraction(float(ro[-1])) - exact) <= 2 ** 5 * (k + 1) * unit + abs(exact) / 2 ** 53


def test_special_values(dump):
    tiny, big = 2.0 ** -1070, 2.0 ** 1023
    out = dump(np.full((5, 2), 0.5), np.array([[0.0, 0.0], [tiny, tiny], [np.inf, 1.0], [np.nan, 1.0], [big, -big / 2]]))
    assert np.array_equal(out[0], [0, 0, 0]) and np.array_equal(out[1], [0, 0, 0])   # subnormal values count as 0
    assert np.isnan(out[2]).all() and np.isnan(out[3]).all()                        # a block that is not finite
    assert np.array_equal(out[4], [big, -big / 2, big / 4])
