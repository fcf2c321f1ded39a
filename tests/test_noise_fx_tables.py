"""The fixed-point noise's tables (paper_1311_1056_gb300/csrc/noise_fx_tables.cuh) are the output of their
generator and what their definitions say (no GPU needed)."""
import math
import os
import re
import subprocess
import sys
from fractions import Fraction

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_1056_gb300", "csrc")


def test_header_is_the_generator_output():
    out = subprocess.run([sys.executable, os.path.join(CSRC, "noise_fx_tables.py")], capture_output=True, text=True,
                         check=True).stdout
    with open(os.path.join(CSRC, "noise_fx_tables.cuh")) as fh:
        assert out.strip() == fh.read().strip()


def test_values_match_their_definitions():
    with open(os.path.join(CSRC, "noise_fx_tables.cuh")) as fh:
        src = fh.read()
    fold = int(re.search(r"NFX_LN_FOLD = (\d+)", src).group(1))
    ln = [(int(a), int(b)) for a, b in re.findall(r"\{(-?\d+)ll, (-?\d+)ll\}", src)]
    assert len(ln) == 128 and ln[127] == (512, 0)
    for i, (r, v) in enumerate(ln):
        assert abs(v / 2.0 ** 57 - math.log(r / 512)) < 4e-16
        for m in (Fraction(128 + i, 128), Fraction(129 + i, 128)):  # the cell's ends
            t = (m / 2 if i >= fold else m) * r / 512 - 1
            assert abs(t) <= Fraction(1, 128)  # the range of the series in the kernel
    sc = [tuple(int(x) for x in q) for q in re.findall(r"\{(-?\d+), (-?\d+), (-?\d+), (-?\d+)\}", src)]
    assert len(sc) == 129
    for j, (ls, hs, lc, hc) in enumerate(sc):
        s, c = (hs * 2 ** 30 + ls) / 2 ** 60, (hc * 2 ** 30 + lc) / 2 ** 60
        assert abs(s - math.sin(math.pi * j / 64)) < 1e-15 and abs(c - math.cos(math.pi * j / 64)) < 1e-15
        assert max(abs(ls), abs(lc)) <= 2 ** 29
