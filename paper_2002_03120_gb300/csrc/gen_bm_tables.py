"""Writes bm_tables.cuh: the constant tables of the table-driven FP64
Box-Muller transform of the GPU pair kernels (correctly rounded doubles,
computed with mpmath at 60 digits).

  LOG_TAB[j]  = { -2 ln c_j, 1 / (1 + j/2048) }                   j = 0..2047
                c_j = 1 + j/2048 in the lower half, (1 + j/2048) / 2 in the upper
  LOG_E[e]    = -2 (e - 24) ln 2                                  e = 0..31
  SC_HI[h]    = { sin(pi/2 h/1024), cos(pi/2 h/1024) }             h = 0..1023
  SC_LO[l]    = { sin, cos of pi/2 (2 l + 1) / 2^22 }              l = 0..2047

Run:  python gen_bm_tables.py  (in this directory)
"""
import os

import mpmath

mpmath.mp.dps = 60


def d(x) -> str:
    return repr(float(x))


def main():
    lines = ["// Generated by gen_bm_tables.py; do not edit.",
             "// Tables of the table-driven FP64 Box-Muller transform (correctly rounded).",
             "#pragma once", ""]

    def table(decl, rows):
        lines.append(decl + " = {")
        lines.extend("    " + r + "," for r in rows)
        lines.append("};")

    c = [1 + mpmath.mpf(j) / 2048 for j in range(2048)]
    table("static __device__ const double2 BM_LOG_TAB[2048]", [f"{{{d(-2 * mpmath.log(x if j < 1024 else x / 2))}, {d(1 / x)}}}" for j, x in enumerate(c)])
    table("static __device__ const double BM_LOG_E[32]", [d(-2 * (e - 24) * mpmath.log(2)) for e in range(32)])
    hi = [mpmath.pi / 2 * h / 1024 for h in range(1024)]
    lo = [mpmath.pi / 2 * (2 * k + 1) / 2 ** 22 for k in range(2048)]
    table("static __device__ const double2 BM_SC_HI[1024]", [f"{{{d(mpmath.sin(x))}, {d(mpmath.cos(x))}}}" for x in hi])
    table("static __device__ const double2 BM_SC_LO[2048]", [f"{{{d(mpmath.sin(x))}, {d(mpmath.cos(x))}}}" for x in lo])
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "bm_tables.cuh")
    with open(out, "w") as f:
        f.write("\n".join(lines) + "\n")


if __name__ == "__main__":
    main()
