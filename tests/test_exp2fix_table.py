"""The table and the polynomial of the fixed-point 2^x (exp2fix_table.inc)
against a 60-digit evaluation."""
import os
import re
from decimal import Decimal, getcontext

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_07094_gb300", "csrc")


def test_exp2fix_constants():
    getcontext().prec = 60
    src = open(os.path.join(CSRC, "exp2fix_table.inc")).read()
    tab = [int(v, 16) for v in re.findall(r"0x([0-9a-f]{16})ull,", src)]
    c = {k: int(v, 16) for k, v in re.findall(r"(EXP2FIX_\w+) = 0x([0-9a-f]+)ull;", src)}
    ln2 = Decimal(2).ln()
    assert len(tab) == 256
    for j, t in enumerate(tab):
        assert abs(Decimal(t) - (Decimal(j) / 256 * ln2).exp() * 2 ** 63) <= Decimal("0.5")
    assert abs(Decimal(c["EXP2FIX_LOG2E_HALF"]) - 2 ** 63 / ln2) <= Decimal("0.5")
    a = [Decimal(c["EXP2FIX_A1"]) / 2 ** 72, Decimal(c["EXP2FIX_A2"]) / 2 ** 82, Decimal(c["EXP2FIX_A3"]) / 2 ** 60,
         Decimal(c["EXP2FIX_A4"]) / 2 ** 60]
    for i in range(257):
        g = Decimal(i) / 256
        p = g * (a[0] + g * (a[1] + g * (a[2] + g * a[3])))
        assert abs(p + 1 - (g / 256 * ln2).exp()) < Decimal(2) ** -56
