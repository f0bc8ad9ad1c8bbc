"""The integer split behind the FP64 tensor-core contractions, in numpy: the
digits reproduce the rounded operands, a chunk's sums stay exact in FP32, and the
kept products carry a dot product to FP64 accuracy."""
from fractions import Fraction

import numpy as np
import pytest

S, BETA, CHUNK = 8, 7, 384


def digits(row):
    """(8 digits per value, exponent): x ~ 2^e sum_i d_i 2^(-7 i), i = 1..8."""
    e = int(np.frexp(np.max(np.abs(row)))[1])
    out = np.zeros((S, row.size), np.int64)
    q = np.array([round(Fraction(float(x)) * Fraction(2) ** (S * BETA - e)) for x in row], dtype=object)
    for i in range(S - 1, 0, -1):
        d = np.array([((int(v) & 127) ^ 64) - 64 for v in q], dtype=object)
        out[i] = d.astype(np.int64)
        q = np.array([(int(v) - int(w)) >> BETA for v, w in zip(q, d)], dtype=object)
    out[0] = q.astype(np.int64)
    return out, e


@pytest.mark.parametrize("spread", [0.0, 6.0, 30.0])
def test_split_dot_is_fp64_accurate(spread):
    rng = np.random.default_rng(int(spread))
    K = 300
    for _ in range(20):
        a = rng.standard_normal(K) * np.exp(-spread * rng.random(K))
        b = rng.standard_normal(K) * np.exp(-spread * np.arange(K) / K)
        da, ea = digits(a)
        db, eb = digits(b)
        assert np.abs(da).max() <= 128 and np.abs(da[1:]).max() <= 64
        got = Fraction(0)
        for c in range(2, S + 2):
            v = sum(int(da[i - 1] @ db[c - i - 1]) for i in range(max(1, c - S), min(S, c - 1) + 1))
            got += Fraction(v) * Fraction(2) ** (ea + eb - BETA * c)
        want = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
        # operands rounded at 2^-57 of their row's scale 2^e, products below
        # c = 10 dropped (7 pairs of digits <= 64 at 2^-70)
        scale = Fraction(2) ** (ea + eb)
        bound = scale * K * (2 * Fraction(1, 2 ** 57) + 8 * 64 * 64 * Fraction(1, 2 ** 70))
        assert abs(got - want) <= bound


def test_chunk_sums_are_exact_in_fp32():
    per_step = max(sum((128 if i == 1 else 64) * (128 if c - i == 1 else 64) for i in range(1, S + 1) if 1 <= c - i <= S)
                   for c in range(2, S + 2))
    assert per_step * CHUNK < 2 ** 24
