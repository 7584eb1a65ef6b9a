"""The single-precision steps by which the kernels find a zero point's exponent and value, against the definition in fractions: a sum of two
halves has more bits than a float, and is rounded up."""
import itertools
import random
import re
from fractions import Fraction

import numpy as np
import pytest


def half(bits):
    return Fraction(float(np.array([min(bits, 0x7BFF)], np.uint16).view(np.float16)[0]))


def rounded_up(x):
    f = np.float32(float(x))                                    # (at most 41 bits: exact in a double)
    if Fraction(float(f)) < x:
        f = np.nextafter(f, np.float32(np.inf))
    else:
        below = np.nextafter(f, np.float32(-np.inf))
        f = below if Fraction(float(below)) >= x else f
    return f


def steps(hi, lo, bits):
    least = half(lo)
    pattern = int(np.array([rounded_up(half(hi) + least)], np.float32).view(np.int32)[0])
    full = ((1 << (bits - 1)) - 1) << (24 - bits)
    e = (pattern >> 23) - 127 - (bits - 1) + ((pattern & 0x7FFFFF) > full) if pattern else 0
    scaled = least / Fraction(2) ** e
    assert Fraction(float(np.float32(float(scaled)))) == scaled          # exact in single precision
    return e, min(int(np.rint(float(scaled))), (1 << bits) - 1)


def definition(hi, lo, bits):
    span, top = half(hi) + half(lo), (1 << bits) - 1
    if span == 0:
        return 0, 0
    e = -40
    while top * Fraction(2) ** e < span:
        e += 1
    return e, min(max(round(half(lo) / Fraction(2) ** e), 0), top)


@pytest.mark.parametrize("bits", [4, 8])
def test_steps_are_the_definition(bits):
    r = random.Random(bits)
    edges = [0, 1, 2, 0x3FF, 0x400, 0x401, 0x3BFF, 0x3C00, 0x4B80, 0x4B81, 0x5BF8, 0x5BF9, 0x7B80, 0x7BF8, 0x7BFF, 0x7C00]
    for hi, lo in itertools.product(edges + [r.randrange(0x7C01) for _ in range(60)], repeat=2):
        assert steps(hi, lo, bits) == definition(hi, lo, bits), (hex(hi), hex(lo))


def test_the_kernels_take_these_steps():
    import os
    path = os.path.join(os.path.dirname(__file__), "..", "paper_2312_05693_b200", "csrc", "aq_quant_math.cuh")
    code = re.sub(r"//[^\n]*", "", open(path).read())
    body = code[code.index("void zero_point_scale("):]
    body = body[:body.index("\n}\n")]
    assert "__fadd_ru(" in body and "__float2int_rn(" in body and "long long" not in body and "double" not in body
