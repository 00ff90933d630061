"""Writes line_lengths.h: the half lengths of the mixed-radix transforms (mixed_fft.cuh),
their radices, and the shared-memory strides of a stored line.

A line is stored at k1 P1 + k2 P2 + k3 in its parity block, the odd block at OFF, lines LS
apart.  The strides are searched: every access pattern of the passes, of the multiply and of
the x passes' untangling is counted in wavefronts (16 banks of 8 bytes per half-warp, 8 banks
of 16 bytes per quarter-warp), and the strides with the fewest, then the shortest line, are
kept.  Two-pass lengths come out free of conflicts, three-pass ones within about 25 %.
Run: python paper_2008_02478_gb300/csrc/gen_lengths.py"""
import multiprocessing
import os

HERE = os.path.dirname(os.path.abspath(__file__))
FINE = [(2, 1, 1), (3, 1, 1), (4, 1, 1), (5, 1, 1), (6, 1, 1), (8, 1, 1), (2, 5, 1), (3, 4, 1), (4, 4, 1), (4, 5, 1),
        (4, 6, 1), (4, 8, 1), (5, 8, 1), (6, 8, 1), (8, 8, 1), (8, 10, 1), (8, 12, 1), (5, 3, 8), (4, 4, 8), (5, 4, 8),
        (6, 4, 8), (6, 5, 8), (4, 8, 8), (5, 8, 8), (6, 8, 8), (6, 10, 8), (8, 8, 8), (8, 10, 8), (8, 12, 8),
        (8, 12, 10), (8, 8, 16), (8, 10, 16), (8, 12, 16), (8, 16, 16)]
COARSE = [(10, 12, 1), (8, 16, 1), (10, 16, 1), (12, 16, 1), (12, 20, 1), (16, 16, 1), (16, 20, 1), (16, 24, 1),
          (20, 24, 1), (16, 32, 1), (20, 32, 1), (24, 32, 1)]


def waves(addrs, banks):
    total = 0
    for g in range(0, 32, banks):
        rows = {}
        for a in set(addrs[g:g + banks]):
            rows.setdefault(a % banks, []).append(a)
        total += max(len(v) for v in rows.values())
    return total


def cost(r1, r2, r3, P2, P1, OFF, LS, banks, lines=8):
    """Wavefronts over what conflict-free accesses take."""
    S1, S2, H = r2 * r3, r3, r1 * r2 * r3
    got = best = 0.0

    def pattern(n, at, weight):
        nonlocal got, best
        starts = list(range(0, max(n - 31, 1), 32))
        for w in starts[::max(1, len(starts) // 4)]:
            got += waves([at(min(i, n - 1)) for i in range(w, w + 32)], banks) * weight / len(starts[::max(1, len(starts) // 4)])
            best += 32 / banks * weight / len(starts[::max(1, len(starts) // 4)])

    def line(i):
        return (i >> 1) * LS + (i & 1) * OFF

    pattern(lines * S1, lambda i: i // S1 * LS + i % S1 // S2 * P2 + i % S2, 2.0)
    if r2 > 1:
        pattern(2 * lines * r1 * S2, lambda i: line(i // S2 // r1) + i // S2 % r1 * P1 + i % S2, 4.0)
    if r3 > 1:
        pattern(2 * lines * r1 * r2, lambda i: line(i // r2 // r1) + i // r2 % r1 * P1 + i % r2 * P2, 4.0)

    def pos(b):
        k = b >> 1
        return (b & 1) * OFF + k % r1 * P1 + k // r1 % r2 * P2 + k // (r1 * r2)

    for b in range(0, H, max(1, H // 6)):  # the multiply: 8 bins and their mirror images
        got += waves([pos(b // 8 * 8 + (i & 15) // 2 if i < 16 else 2 * H - 1 - b // 8 * 8 - (i & 15) // 2) for i in range(32)], banks) * 2 / 6
        best += 32 / banks * 2 / 6
        got += waves([i % 8 * LS + pos((b + i // 8) % (2 * H)) for i in range(32)], banks) / 6  # untangling
        best += 32 / banks / 6
    return got / best


def search(job):
    r1, r2, r3, banks = job
    found = None
    for P2 in ([1] if r3 == 1 else range(r3, r3 + 3)):
        block = (r2 - 1) * P2 + r3
        for P1 in ([1] if r2 == 1 else range(block, block + 9)):
            for o in range(banks):
                OFF = r1 * P1
                while OFF % banks != o:
                    OFF += 1
                for l in range(banks):
                    LS = OFF + r1 * P1
                    while LS % banks != l:
                        LS += 1
                    key = (round(cost(r1, r2, r3, P2, P1, OFF, LS, banks), 2), LS)
                    if found is None or key < found[0]:
                        found = (key, (P2, P1, OFF, LS))
    return found


def main():
    radices = FINE + COARSE
    with multiprocessing.Pool() as pool:
        got = pool.map(search, [(*r, b) for r in radices for b in (16, 8)], chunksize=1)
    out = ["// Generated by gen_lengths.py: X(id, r1, r2, r3, strides of 8-byte values, strides of 16-byte values),",
           "// strides = P2, P1, OFF, LS.", "#pragma once", ""]
    for name, base, part in (("FINE", 0, FINE), ("COARSE", len(FINE), COARSE)):
        out.append("#define BORIS_LENGTHS_%s(X) \\" % name)
        rows = []
        for i, r in enumerate(part):
            f, d = got[2 * (base + i)], got[2 * (base + i) + 1]
            print(r, f, d)
            rows.append("    X(%d, %d, %d, %d, %s, %s)" % (base + i, *r, ", ".join(map(str, f[1])), ", ".join(map(str, d[1]))))
        out.append(" \\\n".join(rows))
        out.append("")
    out += ["#define BORIS_LENGTHS(X) BORIS_LENGTHS_FINE(X) BORIS_LENGTHS_COARSE(X)", "",
            "namespace boris {", "constexpr int N_FINE = %d, N_LENGTHS = %d;" % (len(FINE), len(radices)), "}  // namespace boris"]
    with open(os.path.join(HERE, "line_lengths.h"), "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
