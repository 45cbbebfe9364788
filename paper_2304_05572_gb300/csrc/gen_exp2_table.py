"""Generates exp2_table.inc: 2^(-j/64), j = 0..63, as integers in units of 2^-63 (for the
fixed-point exponential of hgks_fixed.cuh).  Computed in 40-digit arithmetic (mpmath)."""
import os

import mpmath as mp

mp.mp.dps = 40
rows = [int(mp.nint(mp.mpf(2) ** (63 - mp.mpf(j) / 64))) for j in range(64)]
path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "exp2_table.inc")
with open(path, "w") as f:
    f.write("// 2^(-j/64) in units of 2^-63; generated by gen_exp2_table.py\n#define HGKS_EXP2_TABLE { \\\n")
    for k in range(0, 64, 4):
        f.write("    " + ", ".join("0x%016XULL" % v for v in rows[k:k + 4]) + (", \\\n" if k < 60 else " }\n"))
