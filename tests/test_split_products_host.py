"""The split of FP32 values into bf16 planes and the products the contraction keeps, emulated in
numpy: three planes rounded to nearest are the value exactly (24 bits in 8 + 8 + 8), over the
exponents where the third plane is a normal number; the six products with at most two steps down
leave 2^-24 of a product (mid lo + lo mid <= 2 * 2^-8 * 2^-17, lo lo 2^-34 beside it), the three
of two planes 2^-15 (2 * 2^-17 of the planes left out, lo lo 2^-16), whatever the operands' exponents."""
import numpy as np


def _bf16(v):
    b = v.astype(np.float32).view(np.uint32).astype(np.uint64)
    b = ((b + 0x7FFF + ((b >> 16) & 1)) >> 16 << 16).astype(np.uint32)     # to nearest, ties to even
    return b.view(np.float32)


def _planes(v, n):
    out = []
    for _ in range(n):
        h = _bf16(v)
        out.append(h.astype(np.float64))
        v = (v - h).astype(np.float32)
    return out, v


def _values(seed, n=400000):
    rng = np.random.default_rng(seed)
    v = rng.uniform(1.0, 2.0, n).astype(np.float32)
    edge = np.array([1.0, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -23, 1.0 + 2.0 ** -8, 1.0 + 2.0 ** -9, 1.0 + 2.0 ** -12 + 2.0 ** -23,
                     1.0 + 2.0 ** -8 + 2.0 ** -17, 1.998046875], np.float32)
    v = np.concatenate([v, np.repeat(edge, 64)])
    return (v * rng.choice([-1.0, 1.0], len(v)) * 2.0 ** rng.integers(-60, 60, len(v))).astype(np.float32)


def test_three_planes_hold_an_fp32_value():
    v = _values(1)
    p, rest = _planes(v, 3)
    assert np.all(rest == 0) and np.all(p[0] + p[1] + p[2] == v.astype(np.float64))
    assert np.all(np.abs(p[1]) <= 2.0 ** -8 * np.abs(v)) and np.all(np.abs(p[2]) <= 2.0 ** -16 * np.abs(v))


def test_products_kept():
    a, b = _values(2), _values(3)
    exact = a.astype(np.float64) * b.astype(np.float64)
    A, B = _planes(a, 3)[0], _planes(b, 3)[0]
    six = sum(A[i] * B[j] for i in range(3) for j in range(3) if i + j <= 2)
    assert np.max(np.abs(six - exact) / np.abs(exact)) <= 2.0 ** -24 * (1 + 2.0 ** -8)
    three = A[0] * B[0] + A[0] * B[1] + A[1] * B[0]
    assert np.max(np.abs(three - exact) / np.abs(exact)) <= 2.0 ** -15 * (1 + 2.0 ** -8)
