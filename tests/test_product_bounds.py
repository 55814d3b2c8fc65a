"""How large a Montgomery product is before its last subtraction: an integer
model of the steps of mont_mul_pairs (csrc/modexp_core.cuh), with and without
the ring, against the bounds that its comment states."""
import random

import pytest

M64 = (1 << 64) - 1


def _product(a, y, N, S, ring):
    """T before the last subtraction, for S limbs."""
    k = -pow(N, -1, 1 << 64) % (1 << 64)
    F = (k * N + 1) >> 64
    if ring:
        F = (1 << 32 * (S - 2)) + (F - (1 << 32 * (S - 2))) % N
    words = [(y >> 64 * i) & M64 for i in range(S // 2)]
    T = a * words[0]
    for w in words[1:-1]:
        T = (T >> 64) + (T & M64) * F + a * w
    T = (T + (T * k & M64) * N) >> 64
    T += a * words[-1]
    return (T + (T * k & M64) * N) >> 64


def _moduli(S, rng):
    R = 1 << 32 * S
    yield from (R - 1, R - 3, R - (15 << 32 * (S - 2)) + 1, R - (17 << 32 * (S - 2)) + 1)
    yield from ((3 << 32 * S - 2) + 1, (1 << 32 * S - 1) + 1)
    for _ in range(6):
        yield rng.getrandbits(32 * S) | (1 << 32 * S - 1) | 1


@pytest.mark.parametrize("S", (6, 8, 16, 64))
def test_product_bounds(S):
    rng = random.Random(S)
    R = 1 << 32 * S
    for N in _moduli(S, rng):
        tight = N >> 32 * (S - 2) >= (1 << 64) - 16
        below = [0, 1, N - 1, N - 2, N >> 1, *(rng.randrange(N) for _ in range(4))]
        above = [N, R - 1, R - 2, *(rng.randrange(N, R) if N < R else N for _ in range(4))]
        for ring in (False, True):
            for y in below:
                for a in below + above:
                    T = _product(a, y, N, S, ring)
                    assert (T * R - a * y) % N == 0
                    assert T * R < a * y + N * (R + R * 201 // (100 << 64))
                    if tight or a < N:
                        assert T < (3 if tight else 2) * N


def test_a_piece_that_reaches_twice_its_prime():
    """R^2 mod P is within P / 2^70 of P: the product of a piece near R is not
    canonical after one subtraction, those of its residue and of the result are."""
    P = 0xffffffffffffff743130b7c068977c522e54d16e002a9cee4a57be849a4d738f
    y = (1 << 512) % P
    for x in (0xffffffffffffffffff29df9fe921fc384358c97d7f6ca1df9c3587e83519a173,
              0xffffffffffffffffffea44a69711fed6adac385e9905384e8359ccbd3facead2):
        for ring in (False, True):
            T = _product(x, y, P, 8, ring)
            assert 2 * P <= T and (T - P << 64) < P * ((1 << 64) + 3)
            assert _product(x % P, y, P, 8, ring) < 2 * P
            assert _product(T - P, T - P, P, 8, ring) < 2 * P
            assert _product(T - P, 1, P, 8, ring) < 2 * P
