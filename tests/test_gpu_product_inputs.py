"""Products of pieces that are not below their modulus.  The CRT kernels take
a chunk in pieces of one prime's width, and a low piece is any value below
2^(32 S), not below the prime.  The prime P was built so that R^2 mod P is
within P / 2^70 of P; for a low piece near R the product with it then reaches
2P, which one subtraction does not bring below P."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NBITS = 512
P0 = 0xffffffffffffff743130b7c068977c522e54d16e002a9cee4a57be849a4d738f
Q0 = 0xfffffffffffffffffffffffffffffffffffffffffffffffffffffffffffffdb5
# Multiples of P0 below P0 Q0 whose pieces' products are P0 + t and P0 - t with t > 0.
MULTIPLES = (
    0x540f0a6bf7f7582eb9777ae688c1952ab66707e7ddcd851ed4d632b71f6e32e9ffffffffffffffffff29df9fe921fc384358c97d7f6ca1df9c3587e83519a173,
    0x596192ca971be6499d2cfc7127294d230ea3555390bcb1b82dbc5070b97f673dffffffffffffffffffea44a69711fed6adac385e9905384e8359ccbd3facead2,
    0xbec849c776132797bca88f301b203fcff3c9aea97b67102ade81c63c0efa4989ffffffffffffffffff06435af3efe58c361ebe71c0faada024891e988de29d49,
    0xcbfd82fc2076cc24eb6506b13dd4adffc69ed217546b1d9ccac38054096666ffffffffffffffffffff66a50b33bcf3a3adff2ff2db9256c3eebf55eb0b1d7e1,
)


def _limbs(values, nbits):
    raw = b"".join(v.to_bytes(nbits // 8, "little") for v in values)
    return np.frombuffer(raw, np.uint32).reshape(len(values), nbits // 32).copy()


def _device(values):
    import torch

    return torch.from_numpy(_limbs(values, NBITS).view(np.int32)).cuda()


@pytest.fixture(scope="module")
def env():
    import paper_2111_11924_gb300 as P

    ctx = P.Context(0)
    ks = ctx.keyset_from_primes(NBITS, 65537, _limbs([P0], NBITS // 2), _limbs([Q0], NBITS // 2))
    yield P, ctx, ks
    ks.free()
    ctx.close()


@pytest.mark.parametrize("use_crt", (True, False))
def test_blinding_value_that_shares_a_prime(env, use_crt):
    P, ctx, ks = env
    N = P0 * Q0
    assert all(v % P0 == 0 and v < N for v in MULTIPLES)
    for i, v in enumerate(MULTIPLES):
        cr = [3, 5, 7, 11, 13]
        cr[i] = v
        ctx.decrypt_blinded(ks, _device([2] * 5), _device(cr), use_crt=use_crt)
        code, first = ctx.status_detail()
        assert (code, first) == (P.pmkrsa.PMK_ENOINV, i), i


def test_low_pieces_near_the_top(env):
    """The same values as ciphertexts: the result is still the exact power."""
    import torch

    P, ctx, ks = env
    N = P0 * Q0
    d = pow(65537, -1, (P0 - 1) * (Q0 - 1))
    rng = np.random.default_rng(7)
    low = (1 << NBITS // 2) - 1
    c = [*MULTIPLES, *(v ^ (1 << NBITS // 2) for v in MULTIPLES)]
    c += [int.from_bytes(rng.bytes(NBITS // 8), "little") % N | low for _ in range(8)]
    c = [v % N for v in c]
    want = _device([pow(v, d, N) for v in c])
    for use_crt in (False, True):
        assert torch.equal(ctx.decrypt_chunks(ks, _device(c), use_crt=use_crt), want), use_crt
    r = [pow(17 + i, 65537, N) for i in range(len(c))]
    star = [v * x % N for v, x in zip(c, r)]
    for use_crt in (False, True):
        assert torch.equal(ctx.decrypt_blinded(ks, _device(star), _device(r), use_crt=use_crt), want), use_crt
    ctx.check()
