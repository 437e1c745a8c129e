"""The balanced digit slices of the float64 block products (csrc/dm_slices.cuh), restated in exact integers.

S = 7 digits in base 2^8 (K <= 128) or S = 8 in base 2^7 (K <= 512): every digit is exact in bf16, the digits
give the operand to half of 2^(e-55), every accumulator stays within 2^24, and the products with
s + t <= S + 2 give the exact product to the bound of the dropped ones."""
from fractions import Fraction

import numpy as np
import pytest


def digits(v, e, S):
    """Integers d_1 .. d_S with v = 2^(e+1) sum d_s base^-s up to the rounding."""
    bits = 8 if S == 7 else 7
    y = Fraction(v) * Fraction(2) ** (55 - e)
    Y = int(abs(y) + Fraction(1, 2)) * (1 if y >= 0 else -1)
    half, Z = 1 << (bits - 1), Y + sum((1 << (bits - 1)) << (bits * i) for i in range(S))
    out = [(Z >> (bits * (S - 1))) - half]
    out += [((Z >> (bits * (S - 1 - i))) & ((1 << bits) - 1)) - half for i in range(1, S)]
    return out


def values():
    rng = np.random.default_rng(5)
    v = list(rng.uniform(-1, 1, 200)) + [0.0, 1 - 2.0**-53, -(1 - 2.0**-53), 0.5, -0.5, 2.0**-60, -(2.0**-54), 2.0**-1022]
    return v + list(rng.uniform(-1, 1, 50) * 2.0 ** rng.integers(-70, 0, 50))


@pytest.mark.parametrize("S", [7, 8])
def test_digits_are_exact_in_bf16_and_give_the_value(S):
    bits = 8 if S == 7 else 7
    for v in values():
        d = digits(v, 0, S)
        assert all(abs(x) <= 1 << (bits - 1) for x in d)  # at most 2^7: bf16 holds every integer to 2^8
        back = 2 * sum(Fraction(x, 1 << (bits * (s + 1))) for s, x in enumerate(d))
        assert abs(back - Fraction(v)) <= Fraction(1, 2**56)


@pytest.mark.parametrize("S,K", [(7, 32), (7, 128), (8, 256), (8, 512)])
def test_accumulators_and_product(S, K):
    bits = 8 if S == 7 else 7
    pairs = {d: [(s, d - s) for s in range(1, S + 1) if 1 <= d - s <= S] for d in range(2, S + 3)}
    assert max(len(p) for p in pairs.values()) * K * (1 << (2 * bits - 2)) <= 1 << 24
    rng = np.random.default_rng(K)
    L, R = rng.uniform(-1, 1, K), rng.uniform(-1, 1, K)
    DL, DR = [digits(v, 0, S) for v in L], [digits(v, 0, S) for v in R]
    acc = {d: sum(DL[k][s - 1] * DR[k][t - 1] for k in range(K) for s, t in p) for d, p in pairs.items()}
    assert all(abs(a) <= 1 << 24 for a in acc.values())
    got = 4 * sum(Fraction(a, 1 << (bits * d)) for d, a in acc.items())
    exact = sum(Fraction(a) * Fraction(b) for a, b in zip(L, R))
    # operands rounded at 2^-56 each, and the dropped pairs: those of s + t = S + 3 at most (S - 2) 2^(2 bits
    # - 2) base^-(S+3) per term, the rest less than as much again
    dropped = Fraction(4 * 2 * (S - 2) << (2 * bits - 2), 1 << (bits * (S + 3)))
    assert abs(got - exact) <= K * (Fraction(2, 2**56) + dropped)
