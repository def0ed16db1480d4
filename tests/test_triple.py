"""The three-float arithmetic of the mixed solver's state on the host against exact rationals, and the
same bits on the device.

Bounds, relative to the larger operand or the product: what a sum or product of numbers of three floats
drops is the rounding of its last part (2^-24 of a part of at most 2^-47) and of the few terms that go
into it, below 2^-68; a product with a number of two floats keeps two floats (2^-46)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc


def operands(n, seed, kind):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(n) * 2.0 ** rng.integers(-12, 1, n)
    y = rng.standard_normal(n) * 2.0 ** rng.integers(-30, 1, n)
    if kind == "increments":
        y = x * rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-40, 1, n)
    if kind == "cancelling":
        y = -x * (1.0 + rng.standard_normal(n) * 2.0 ** rng.integers(-50, 0, n).astype(float))
    if kind == "simple":
        x[:6], y[:6] = [0.0, 1.0, 1.0, -0.5, 0.0, 1.0], [0.0, -1.0, 2.0 ** -53, 0.5, 1.0, 0.0]
    return x, y


def exact(t):
    return [sum((Fraction(float(v)) for v in row), Fraction(0)) for row in t]


@pytest.mark.parametrize("kind", ["random", "increments", "cancelling", "simple"])
def test_host_arithmetic_against_exact_rationals(kind):
    x, y = operands(3000, 11, kind)
    X, Y = [Fraction(v) for v in x], [Fraction(v) for v in y]
    two = [sum((Fraction(float(v)) for v in row[:2]), Fraction(0)) for row in msqoc.selftest_triple("split", y, y)]
    assert exact(msqoc.selftest_triple("split", x, y)) == X
    assert exact(msqoc.selftest_triple("round", x, y)) == X
    ops = {"add3": (lambda a, b, t: a + b, 68), "sum": (lambda a, b, t: a + b, 68), "mul": (lambda a, b, t: a * b, 68),
           "kappa": (lambda a, b, t: a * t, 46)}
    if kind == "increments":
        ops["add"] = (lambda a, b, t: a + t, 68)
    for op, (f, bits) in ops.items():
        got = exact(msqoc.selftest_triple(op, x, y))
        for g, a, b, t in zip(got, X, Y, two):
            size = abs(a * b) if op in ("mul", "kappa") else max(abs(a), abs(b))
            assert abs(g - f(a, b, t)) <= size * Fraction(1, 2 ** bits), (op, float(a), float(b))


@pytest.mark.gpu
@pytest.mark.parametrize("op", msqoc.TRIPLE_OPS)
def test_device_gives_the_same_bits(op):
    for kind in ("random", "increments", "cancelling", "simple"):
        x, y = operands(5000, 12, kind)
        h, d = (msqoc.selftest_triple(op, x, y, device=dev) for dev in (False, True))
        np.testing.assert_array_equal(h.view(np.uint32), d.view(np.uint32))
