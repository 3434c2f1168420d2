"""Tables of e^{-j/256}, j = 0..511, for the opaque segments of the FP64 table march; writes ``exp_table.h``
next to this script.

The march takes e^{-x} for x >= 2 as e^{-2m} e^{-j/256} e^{-r} with x = 2 m + j / 256 + r and
|r| <= 1/512; the middle factor comes from here, the value of the exponential series in 40-digit
arithmetic rounded to double, and what that rounding left out, relative to it, as a float (C99
hexadecimal literals).

    python paper_2512_12466_gb300/csrc/gen_exp_table.py
"""
import os
import struct

import mpmath as mp

STEPS = 512
HERE = os.path.dirname(os.path.abspath(__file__))


def exp_minus(y):
    s = term = mp.mpf(1)
    n = 0
    while abs(term) > mp.mpf(10) ** -38:
        n += 1
        term *= -y / n
        s += term
    return s


def rows():
    mp.mp.dps = 40
    exact = [exp_minus(mp.mpf(j) / 256) for j in range(STEPS)]
    return [(float(v), struct.unpack("<f", struct.pack("<f", float(v / mp.mpf(float(v)) - 1)))[0]) for v in exact]


def write(path=os.path.join(HERE, "exp_table.h")):
    lines = [
        "// Generated by gen_exp_table.py: e^{-j/256}, j = 0..511, rounded to double, and the part that",
        "// rounding left out, relative to it.",
        "#pragma once",
        "",
        "namespace nyx {",
    ]
    v = rows()
    for name, kind, k, per in (("kExpFrac", "double", 0, 4), ("kExpFracRest", "float", 1, 6)):
        lines.append(f"__device__ const {kind} {name}[{STEPS}] = {{")
        for j in range(0, STEPS, per):
            lines.append("    " + ", ".join(x[k].hex() + ("f" if k else "") for x in v[j:j + per]) + ",")
        lines.append("};")
    lines += ["}  // namespace nyx", ""]
    with open(path, "w") as f:
        f.write("\n".join(lines))


if __name__ == "__main__":
    write()
