"""The Montgomery product at the edges of its carries: moduli and operands
whose limbs are nearly all ones, so that every carry chain, the words held
back above a lane's limbs and the lane-to-lane lookahead run over, through
every compiled geometry (2 to 16 limbs per lane, 2 to 32 lanes).  Integers are
compared with Python's pow, exactly."""
import functools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _limbs(values, nbits):
    raw = b"".join(v.to_bytes(nbits // 8, "little") for v in values)
    return np.frombuffer(raw, np.uint32).reshape(len(values), nbits // 32).copy()


@functools.lru_cache(maxsize=None)
def _top_primes(bits):
    """The two largest primes below 2^bits that are 2 mod 3 (so that e = 3 and
    65537 are usable); Fermat tests to two bases, and the library checks again."""
    found, c = [], (1 << bits) - 1
    small = [p for p in range(3, 2000, 2) if all(p % q for q in range(3, int(p ** 0.5) + 1, 2))]
    while len(found) < 2:
        if c % 3 == 2 and all(c % p for p in small) and pow(2, c - 1, c) == 1 and pow(7, c - 1, c) == 1:
            found.append(c)
        c -= 2
    return found


def _operands(N, nbits, rng):
    ones = (1 << nbits) - 1
    vals = [0, 1, 2, N - 1, N - 2, N >> 1, (N >> 1) + 1, ones >> 1, ones >> 32, ones >> (nbits // 2)]
    for k in range(12):  # runs of ones and zeros of random lengths, then random values
        v, bit = 0, k & 1
        while v.bit_length() < nbits and (bit or v):
            run = int(rng.integers(1, 97))
            v = (v << run) | (((1 << run) - 1) if bit else 0)
            bit ^= 1
        vals.append(v % N)
    vals += [int.from_bytes(rng.bytes(nbits // 8), "little") % N for _ in range(4)]
    return vals


@pytest.mark.parametrize("nbits,crt", [(128, False), (256, False), (512, False), (1024, False), (2048, False),
                                       (3072, False), (256, True), (512, True), (1024, True), (2048, True),
                                       (3072, True)])
def test_all_ones_moduli_every_geometry(nbits, crt):
    import torch

    import paper_2111_11924_gb300 as P

    ctx = P.Context(0)
    p, q = _top_primes(nbits // 2)
    N = p * q
    limbs = nbits // 32 // (2 if crt else 1)
    rng = np.random.default_rng(nbits + crt)
    m = _operands(N, nbits, rng)
    for e in (3, 65537):
        ks = ctx.keyset_from_primes(nbits, e, _limbs([p], nbits // 2), _limbs([q], nbits // 2))
        c = [pow(x, e, N) for x in m]
        d_m = torch.from_numpy(_limbs(m, nbits).view(np.int32)).cuda()
        d_c = torch.from_numpy(_limbs(c, nbits).view(np.int32)).cuda()
        for tpi, form in P.kernel_configs(limbs, crt):
            ctx.set_kernel_config(limbs, crt, tpi, form)
            if not crt:
                assert torch.equal(ctx.encrypt_chunks(ks, d_m), d_c), (tpi, form, e, "encrypt")
            assert torch.equal(ctx.decrypt_chunks(ks, d_c, use_crt=crt), d_m), (tpi, form, e, "decrypt")
        ctx.check()
        ks.free()
    ctx.close()


@pytest.mark.parametrize("nbits", (128, 512, 1024, 2048))
def test_chunks_not_below_the_modulus(nbits):
    """A chunk >= N is reported and still gives its residue's power, per call
    and through the task queues, for every geometry."""
    import torch

    import paper_2111_11924_gb300 as P
    from paper_2111_11924_gb300 import pmkrsa

    ctx = P.Context(0)
    ks = ctx.keygen(2, nbits, 65537, 23)
    Ns = [int.from_bytes(r.tobytes(), "little") for r in ks.export()["N"]]
    top = (1 << nbits) - 1
    m = [x for pair in zip(*((N, N + 1, top, N - 1, 0, 3) for N in Ns)) for x in pair]  # chunk t under key t mod 2
    d_m = torch.from_numpy(_limbs(m, nbits).view(np.int32)).cuda()
    want = torch.from_numpy(_limbs([pow(x, 65537, Ns[t % 2]) for t, x in enumerate(m)], nbits).view(np.int32)).cuda()
    for tpi, form in P.kernel_configs(nbits // 32, False):
        ctx.set_kernel_config(nbits // 32, False, tpi, form)
        assert torch.equal(ctx.encrypt_chunks(ks, d_m), want), (tpi, form)
        assert ctx.status() == pmkrsa.PMK_ERANGE
        for direct in (256, 0):
            out = torch.zeros_like(d_m)
            ctx.set_batch_direct_max(direct)
            batch = ctx.batch([(ks, d_m, out, pmkrsa.OP_ENCRYPT)])
            batch.launch()
            assert ctx.status() == pmkrsa.PMK_ERANGE
            assert torch.equal(out, want), (tpi, form, direct)
    ctx.close()
