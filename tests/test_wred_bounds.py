"""The bound on the division-step inverse (csrc/wred.cuh) and the conversion of its limbs to
packed words, in integers, from the constants in the source."""
import os
import re
from fractions import Fraction

from oracle import fq

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = open(os.path.join(ROOT, "paper_2502_11660_gb300", "csrc", "wred.cuh")).read()
BITS, LIMBS = 27, 15


def table(name):
    body = re.search(name + r"\[16\] = \{([^}]*)\}", SRC).group(1)
    return [int(w) for w in body.split(",")]


def value(limbs):
    return sum(v << (BITS * j) for j, v in enumerate(limbs))


def offset():
    """The multiple of p that the conversion adds to the limbs, its limbs."""
    k = int(re.search(r"l\[j\] \+ k(\d+)P\[j\]", SRC).group(1))
    return k, table(f"k{k}P")


def largest_inverse():
    """The bound on |d| after every round: each adds at most 2^26 p / 2^27, from max(0, 1)."""
    rounds = int(re.search(r"kInvRounds = (\d+)", SRC).group(1))
    assert BITS * rounds >= (45907 * fq.P.bit_length() + 26313) // 19929   # the steps that suffice
    bound = Fraction(1)
    for _ in range(rounds):
        bound += Fraction(fq.P * (1 << 26), 1 << 27)
    return int(bound)


def pack(limbs, add0=0):
    """to_fe_times' carries and packing: twelve words, and whether nothing was lost."""
    _, off = offset()
    words, carry = [0] * 13, add0
    for j in range(LIMBS):
        carry += limbs[j] + off[j]
        dig = carry & ((1 << BITS) - 1)
        carry >>= BITS
        bit = BITS * j
        v = dig << (bit & 31)
        words[bit >> 5] |= v & 0xffffffff
        words[(bit >> 5) + 1] |= v >> 32
    return sum(w << (32 * k) for k, w in enumerate(words[:12])), carry == 0 and words[12] == 0


def split(v):
    """Signed limbs of v, the top one taking what is left."""
    out = []
    for _ in range(LIMBS - 1):
        d = ((v + (1 << (BITS - 1))) & ((1 << BITS) - 1)) - (1 << (BITS - 1))
        out.append(d)
        v = (v - d) >> BITS
    return out + [v]


def test_constants():
    assert value(table("kP27")) == fq.P
    k, off = offset()
    assert value(off) == k * fq.P


def test_every_inverse_converts():
    k, _ = offset()
    b = largest_inverse()
    for v in (-b, -b + 1, -fq.P, -1, 0, 1, fq.P, b - 1, b):
        for add0 in (0, -1):
            packed, whole = pack(split(v), add0)
            assert whole and packed == v + add0 + k * fq.P, (v, add0)
            assert packed * (fq.P - 1) // (1 << 384) + fq.P < 2 * fq.P   # the Montgomery product's range
