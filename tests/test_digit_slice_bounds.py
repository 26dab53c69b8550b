"""The digit-slice kernels' FP32 sums of digit products at their worst: the
sequence's digits 0..255 below a leading one within 64, the other operand's
-128..127 below a leading one within 64, every digit extreme and of one sign,
at the block sizes of the source, added one by one in FP32 and in integers.
What FP32 loses is a small part of the digits that are not kept (2^-54 of the
operands' bounds a term)."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_5299_gb300", "csrc",
                   "legendre_ds.cu")
DIG, ORD = 7, 8


def constant(name):
    return int(re.search(r"constexpr int %s = (\d+);" % name, open(SRC).read()).group(1))


def worst(i, j):
    # odd products, so that a partial sum beyond 2^24 loses its last bit
    return (63 if i == 0 else 255) * (63 if j == 0 else 127)


def sums(products):
    f, n = np.float32(0.0), 0
    for p in products:
        f, n = np.float32(f + np.float32(p)), n + p
    return f, n


def unit(s):
    return 2.0 ** (-8 * s - 12)  # of the operands' bounds


def test_synthesis_orders():
    terms = constant("DSS_KB")
    lost = 0.0
    for s in range(ORD):
        pairs = [(i, s - i) for i in range(DIG) if 0 <= s - i < DIG]
        f, n = sums([worst(i, j) for _ in range(terms) for i, j in pairs])
        if s <= 5:
            assert int(f) == n, (s, n)
            assert terms * sum((64 if i == 0 else 255) * (64 if j == 0 else 128) for i, j in pairs) < 2**24, s
        lost += abs(int(f) - n) * unit(s)
    assert lost < 0.03 * terms * 2.0**-54


def test_adjoint_orders():
    """Accumulator d holds order o = j + d from digits d and d + 4 of the
    sequence and is exact; an order adds up four of them in FP32."""
    terms = constant("DS_PAIRS")
    lost = 0.0
    for o in range(ORD):
        acc = []
        for d in range(min(4, o + 1)):
            pairs = [(i, o - i) for i in (d, d + 4) if i < DIG and 0 <= o - i < DIG]
            f, n = sums([worst(i, j) for _ in range(terms) for i, j in pairs])
            assert int(f) == n, (o, d)
            acc.append((f, n))
        f = acc[0][0]
        for x in acc[1:]:
            f = np.float32(f + x[0])
        n = sum(x[1] for x in acc)
        if o <= 4:
            assert int(f) == n, o
        lost += abs(int(f) - n) * unit(o)
    assert lost < 0.06 * terms * 2.0**-54
