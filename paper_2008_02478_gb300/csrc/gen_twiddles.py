"""Writes twiddle128.h and twiddle480.h: exp(-2 pi i e / N), e in [0, N), N = 128
and 480 (the latter holds every root of unity of the mixed-radix transforms:
480 = 2^5 3 5), from FP64 cos/sin, as literal tables that the in-register
transforms index with compile-time indices (the values fold into the
arithmetic instructions).
Run: python paper_2008_02478_gb300/csrc/gen_twiddles.py"""
import math
import os

HERE = os.path.dirname(os.path.abspath(__file__))


def write(n):
    re = [math.cos(2 * math.pi * e / n) for e in range(n)]
    im = [-math.sin(2 * math.pi * e / n) for e in range(n)]
    fmt = lambda v: repr(float(v))
    lines = ["// Generated by gen_twiddles.py (FP64 cos/sin): w_%d^e = exp(-2 pi i e / %d)." % (n, n),
             "#pragma once", "", "namespace boris {", ""]
    for name, vals in (("w%d_re" % n, re), ("w%d_im" % n, im)):
        lines.append("__host__ __device__ constexpr double %s(int e)" % name)
        lines.append("{")
        lines.append("    constexpr double t[%d] = {" % n)
        for i in range(0, n, 4):
            lines.append("        " + ", ".join(fmt(v) for v in vals[i:i + 4]) + ",")
        lines.append("    };")
        lines.append("    return t[e];")
        lines.append("}")
        lines.append("")
    lines.append("}  // namespace boris")
    with open(os.path.join(HERE, "twiddle%d.h" % n), "w") as f:
        f.write("\n".join(lines) + "\n")


def main():
    write(128)
    write(480)


if __name__ == "__main__":
    main()
