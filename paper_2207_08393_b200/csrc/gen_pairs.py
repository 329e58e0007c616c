"""Writes pairs.def: the phase-encode extents (n1, n2) whose row-tile kernels split both axes into two register
stages with a middle radix of at most 24.  The other extents run the same three passes with one row per block
(single-stage n1), single-stage rows (n2) or a middle radix of 32.

    python paper_2207_08393_b200/csrc/gen_pairs.py        # rewrites pairs.def next to this file
"""
import os
import re

HERE = os.path.dirname(os.path.abspath(__file__))


def plans():
    """{length: (R0, R1)}, the plans of the contiguous axis."""
    text = open(os.path.join(HERE, "sizes.def")).read()
    return {int(n): (int(a0), int(a1)) for n, a0, a1 in re.findall(r"GLEAM_SIZE\((\d+), (\d+), (\d+),", text)}


def main():
    P = plans()
    pairs = [(n1, ry, by, n2, z0) for n2, (z0, z1) in sorted(P.items()) if z1 > 1
             for n1, (ry, by) in sorted(P.items()) if 1 < by <= 24]
    with open(os.path.join(HERE, "pairs.def"), "w") as fh:
        fh.write("// Generated by gen_pairs.py from sizes.def.  GLEAM_PAIR(n1, RY, BY, n2, Z0): n1 = RY * BY, first radix Z0 of n2.\n")
        for p in pairs:
            fh.write("GLEAM_PAIR(%d, %d, %d, %d, %d)\n" % p)
    print(len(pairs), "pairs")


if __name__ == "__main__":
    main()
