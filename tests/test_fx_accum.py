"""The mixed solver's iterate in integer limbs (csrc/fxaccum.cuh) against exact sums: it keeps
its bits over all updates of a refinement (host code, no GPU needed)."""
import os
import struct
import subprocess
from fractions import Fraction

import pytest

from tests.test_fpconv import HERE, _nvcc


def test_iterate_keeps_its_bits(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fx_accum_run")
    subprocess.run([nvcc, "-O2", "-std=c++17", os.path.join(HERE, "native", "fx_accum_run.cu"), "-o", exe], check=True,
                   capture_output=True)
    lines = subprocess.run([exe], capture_output=True, text=True, timeout=600, check=True).stdout.splitlines()
    assert len(lines) == 3000
    for line in lines:
        w = line.split()
        n, scale = int(w[0]), Fraction(struct.unpack("<d", int(w[1], 16).to_bytes(8, "little"))[0])
        e = [Fraction(struct.unpack("<f", int(v, 16).to_bytes(4, "little"))[0]) for v in w[2:26]]
        E, x = int(w[26]), [int(v) for v in w[27:51]]
        if n == 0:
            exact, bound = [Fraction(0)] * 24, Fraction(0)
        exact = [a + scale * b for a, b in zip(exact, e)]
        top = max(abs(v) for v in x)
        assert E > 0 and 2**56 - 1 <= top <= 2**57
        unit = Fraction(2) ** (E - 1079)
        # An update rounds, in units of the new exponent or of half that: the old value once,
        # the product twice, the sum once.  Error of the values before it, which may cancel,
        # counts in full.
        if n == 0 or any(v != 0 for v in e):
            bound += 2 * unit
        assert all(abs(v * unit - a) <= bound for v, a in zip(x, exact)), n
