"""The integer conversions of the digit products, compiled for the host with
undefined shifts and overflows trapped: a recombined sum to binary64
(split_to_double) over zero, ties, carries and the ends of the range, and T's
entries between binary64 and binary32 (f32_of, f64_of).  No GPU."""
import math
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1301_1071_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("split") / "split_scalars")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-Xcompiler", "-fsanitize=shift", "-Xcompiler", "-fsanitize=signed-integer-overflow",
                    "-Xcompiler", "-fsanitize-undefined-trap-on-error", "-I", CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "host", "split_scalars.cu")], check=True, capture_output=True)

    def go(lines):
        r = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, f"ended with {r.returncode} after {len(r.stdout.split())} of {len(lines)}"
        return [int(x) for x in r.stdout.split()]
    return go


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _nearest(P, s):
    """P 2^s rounded to 53 bits, ties away from zero (normal results)."""
    a = abs(P)
    drop = a.bit_length() - 53
    if drop > 0:
        a = (a + (1 << (drop - 1))) >> drop << drop
    return math.copysign(float(Fraction(a) * Fraction(2) ** s), P)


def _sums():
    rng = np.random.default_rng(5)
    P = [0, 1, -1, 2**62, -2**62, 2**63 - 1, -(2**63 - 1), -2**63, 2**53, 2**53 + 1, 2**54 - 1, 2**54 + 2, -(2**54 + 2),
         2**63 - 2**9, 2**63 - 2**9 - 1, 2**62 + 2**8, 2**62 + 2**8 - 1, 2**62 - 1]
    for k in range(1, 63):
        P += [2**k + 1, -(2**k - 1), int(rng.integers(2**(k - 1), 2**k)), -int(rng.integers(2**(k - 1), 2**k))]
    return P


def test_split_to_double(run):
    cases = [(P, s) for P in _sums() for s in (-2100, -1000, -124, -60, 0, 3, 900) if P != 0]
    got = run([f"s {P} {s}" for P, s in cases])
    for (P, s), b in zip(cases, got):
        if s == -2100:  # below the subnormal range
            assert b in (0, 1 << 63), (P, s)
        else:
            assert b == _bits(_nearest(P, s)), (P, s)


def test_split_to_double_zero(run):
    """A zero sum (every padding column, every zero row) is zero at any exponent."""
    exps = [-110000, -5000, -2100, -1085, -1022, -1, 0, 1, 958, 1023, 5000, 1 << 20]
    assert run([f"s 0 {s}" for s in exps]) == [0] * len(exps)


def test_split_to_double_ends(run):
    """Subnormal results within one unit, overflow to infinity."""
    cases = [(P, s) for P in (1, -3, 2**52 + 1, 2**62 - 1) for s in (-1137, -1130, -1100, -1074, -1060)]
    for (P, s), b in zip(cases, run([f"s {P} {s}" for P, s in cases])):
        got = Fraction(struct.unpack("<d", struct.pack("<Q", b))[0])
        want = Fraction(P) * Fraction(2) ** s
        assert abs(got - want) <= max(Fraction(2) ** -1074, abs(want) * Fraction(2) ** -53), (P, s)
    assert run(["s 9223372036854775807 961", "s -4611686018427387904 1000"]) == [_bits(np.inf), _bits(-np.inf)]


def test_f32_of_and_f64_of(run):
    """The same bits as the conversions (NaN: a NaN)."""
    rng = np.random.default_rng(6)
    d = [0.0, -0.0, 1.0, 2.0**-126, 2.0**-127, 2.0**-149, 2.0**-150, 1.5 * 2.0**-150, 2.0**128, 2.0**128 - 2.0**103,
         2.0**128 - 2.0**104, 1 + 2.0**-24, 1 + 3 * 2.0**-24, 1 + 2.0**-24 + 2.0**-52, 2.0**-126 - 2.0**-151,
         2.0**1023, 5e-324, np.inf, -np.inf]
    d += list(rng.standard_normal(500) * 2.0 ** rng.integers(-160, 140, 500))
    got = run([f"d {_bits(float(x))}" for x in d])
    with np.errstate(over="ignore", under="ignore"):
        want = np.array(d, dtype=np.float64).astype(np.float32).view(np.uint32)
    assert got == [int(x) for x in want]
    f = np.concatenate([np.array([0.0, -0.0, 1.0, -1.5, 2.0**-126, 2.0**-149, 3.4e38, np.inf, -np.inf], np.float32),
                        rng.integers(0, 2**32, 500, dtype=np.uint32).view(np.float32)])
    f = f[~np.isnan(f)]
    got = run([f"f {int(x)}" for x in f.view(np.uint32)])
    assert got == [int(x) for x in f.astype(np.float64).view(np.uint64)]
    nan64, nan32 = 0x7FF8000000000000, 0x7FC00000
    assert run([f"d {nan64}"])[0] & 0x7FFFFFFF > 0x7F800000
    assert run([f"f {nan32}"])[0] & ~(1 << 63) > 0x7FF0000000000000
