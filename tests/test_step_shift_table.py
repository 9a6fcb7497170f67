"""bk_cosh_shift.inc is what its generator writes, and moves each step to the one
whose 2 cosh is the rounded entry of bk_cosh_table.inc (Taylor series in exact
rationals, to second order in the shift, about 1e-32)."""
import importlib.util
import os
import re
from fractions import Fraction

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2502_00356_gb300", "csrc")
HEX = re.compile(r"-?0x[01]\.[0-9a-f]+p[+-]\d+")


def parse(inc):
    with open(os.path.join(CSRC, inc)) as f:
        return [float.fromhex(h) for h in HEX.findall(f.read())]


def test_shift_table():
    spec = importlib.util.spec_from_file_location("gen", os.path.join(CSRC, "gen_cosh_table.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    shift, cosh = parse("bk_cosh_shift.inc"), parse("bk_cosh_table.inc")
    assert shift == gen.shifts() and len(shift) == len(cosh) == 3328
    for k in range(0, 3328, 61):
        h = Fraction(2) ** (k // 256 - 12) * (1 + Fraction(k % 256, 256))
        term, c, s, i = Fraction(1), Fraction(0), Fraction(0), 0  # cosh, sinh
        while term > Fraction(1, 2 ** 200):
            c, s = (c + term, s) if i % 2 == 0 else (c, s + term)
            i += 1
            term = term * h / i
        off = float(Fraction(cosh[k]) - 2 * c - 2 * s * Fraction(shift[k]))
        assert abs(off) <= 2.0 ** -24 * abs(float(Fraction(cosh[k]) - 2 * c)) + 1e-31
