"""The nine-bit digits that the split kernels store (csrc/oz_digits.cuh, host-compiled): the digits of
N = round(x 2^(9 s - 1 - E)) in base 512, each exact in BF16, the top one within +-128 and the others
in [-256, 255], and x within half a unit of the last digit."""
import math
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("s", [3, 4, 5, 6, 7])
def test_nine_bit_digits(s, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "oz_digits9_host")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "host", "oz_digits9_host.cu")],
                   check=True, capture_output=True)
    rng = random.Random(s)
    cases = []
    for _ in range(2000):
        c = math.ldexp(0.5 + 0.5 * rng.random(), rng.randint(-900, 900))
        x = rng.choice([c, -c, 0.0, c * rng.uniform(-1, 1), math.ldexp(c, -rng.randrange(60)),
                        -math.ldexp(c * rng.random(), -rng.randrange(60))])
        cases.append((x, c))
    # up to the largest magnitude that an exponent allows (at seven slices the significand is shifted left there)
    for e in (-900, 0, 900):
        c = math.ldexp(1.0 - 2.0 ** -53, e)
        cases += [(sign * math.ldexp(m, e), c) for sign in (1, -1) for k in range(12)
                  for m in (math.ldexp(1.0 - 2.0 ** -53, -k), math.ldexp(0.5, -k), math.ldexp(1.0 - rng.random() * 2.0 ** -40, -k))]
    bits = lambda v: struct.unpack("<Q", struct.pack("<d", v))[0]  # noqa: E731
    inp = "".join(f"{bits(x):016x} {bits(c):016x} {s}\n" for x, c in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout.splitlines()
    for (x, c), line in zip(cases, out):
        d = [struct.unpack("<f", struct.pack("<I", int(h, 16) << 16))[0] for h in line.split()]
        assert len(d) == s and abs(d[0]) <= 128 and all(-256 <= v <= 255 for v in d[1:])
        E = math.frexp(c)[1] + 1
        N = sum(int(v) * 512 ** (s - 1 - i) for i, v in enumerate(d))
        unit = Fraction(2) ** (E - (9 * s - 1))
        assert abs(Fraction(x) - N * unit) <= unit / 2
