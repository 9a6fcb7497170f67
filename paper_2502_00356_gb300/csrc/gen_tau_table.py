"""Write bk_tau_table.inc: e^{j/16}, j = -384..384 (769 entries, index
j + 384), as C hex-float literals.

Each value is computed with 60-digit decimal arithmetic and rounded once to
the nearest double.  The table holds the nodes of the integral that the
Matern writers' per-call tables are built from (bk_entry_table.cuh).

    python paper_2502_00356_gb300/csrc/gen_tau_table.py
"""
from __future__ import annotations

import os
from decimal import Decimal, getcontext

J_MAX = 384


def values() -> list[float]:
    getcontext().prec = 60
    return [float(str((Decimal(j) / 16).exp())) for j in range(-J_MAX, J_MAX + 1)]


def main() -> str:
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "bk_tau_table.inc")
    v = values()
    lines = ["// e^{j/16}, j = -384..384, correctly rounded; written by gen_tau_table.py."]
    for a in range(0, len(v), 4):
        lines.append("    " + ", ".join(x.hex() for x in v[a:a + 4]) + ",")
    with open(out, "w") as f:
        f.write("\n".join(lines) + "\n")
    return out


if __name__ == "__main__":
    print(main())
