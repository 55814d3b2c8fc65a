"""The Montgomery product at the edges of its carries where
test_gpu_product_edges.py does not go: keys of 4096 to 8192 bits, the blinded
kernels, the task queues and recombination over four primes, all with the
largest primes of their width, and the choice of lanes by size above 1024
bits.  Integers are compared with Python's pow, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# 2^bits minus the largest primes that are 2 mod 3 and not 1 mod 65537
OFFSETS = {1024: (179, 1397, 6083, 9497), 1536: (7769, 8333), 2048: (2543, 8507, 9443, 9509), 3072: (47, 2165),
           4096: (2549, 8627)}


def _limbs(values, nbits):
    raw = b"".join(v.to_bytes(nbits // 8, "little") for v in values)
    return np.frombuffer(raw, np.uint32).reshape(len(values), nbits // 32).copy()


def _device(values, nbits):
    import torch

    return torch.from_numpy(_limbs(values, nbits).view(np.int32)).cuda()


def _primes(bits, count=2):
    return [(1 << bits) - o for o in OFFSETS[bits][:count]]


def _operands(N, nbits, rng, randoms=4):
    vals = [0, 1, 2, N - 1, N - 2, N >> 1, (N >> 1) + 1, N >> 32, N >> (nbits // 2), (1 << nbits // 2) - 1,
            N - (1 << nbits // 2)]
    vals += [sum(((1 << 33) - 1) << i for i in range(s, nbits - 34, 67)) % N for s in (0, 31)]  # runs of 33 ones
    return vals + [int.from_bytes(rng.bytes(nbits // 8), "little") % N for _ in range(randoms)]


def _chunks_below(n, nbits, seed):
    import torch

    raw = np.zeros((n, nbits // 8), np.uint8)
    raw[:, :-1] = np.random.default_rng(seed).integers(0, 256, (n, nbits // 8 - 1), dtype=np.uint8)
    return torch.from_numpy(raw.view(np.int32)).cuda()


@pytest.fixture(scope="module")
def env():
    import paper_2111_11924_gb300 as P

    ctx = P.Context(0)
    yield P, ctx
    ctx.close()


@pytest.mark.parametrize("nbits", (2048, 4096, 6144, 8192))
def test_all_ones_moduli_calls_and_queues(env, nbits):
    import torch

    P, ctx = env
    p, q = _primes(nbits // 2)
    ks = ctx.keyset_from_primes(nbits, 65537, _limbs([p], nbits // 2), _limbs([q], nbits // 2))
    m = _operands(p * q, nbits, np.random.default_rng(nbits))
    d_m, d_c = _device(m, nbits), _device([pow(x, 65537, p * q) for x in m], nbits)
    B = P.pmkrsa
    try:
        ctx.set_batch_direct_max(0)
        for limbs, crt in ((nbits // 32, False), (nbits // 64, True)):
            for window in ((5, 4) if crt else (5,)):
                for tpi in sorted({t for t, _ in P.kernel_configs(limbs, crt)}):
                    form = dict(P.kernel_configs(limbs, crt))[tpi]
                    try:
                        ctx.set_kernel_window(limbs, crt, window)
                    except P.PMKError:
                        continue  # no small table at this width
                    ctx.set_kernel_config(limbs, crt, tpi, form)
                    what = (limbs, crt, tpi, window)
                    jobs = [(ks, d_c, torch.zeros_like(d_c), B.OP_DECRYPT_CRT if crt else B.OP_DECRYPT)]
                    if not crt:
                        assert torch.equal(ctx.encrypt_chunks(ks, d_m), d_c), what
                        jobs.append((ks, d_m, torch.zeros_like(d_m), B.OP_ENCRYPT))
                    assert torch.equal(ctx.decrypt_chunks(ks, d_c, use_crt=crt), d_m), what
                    batch = ctx.batch(jobs)
                    assert batch.n_tasks > 0
                    batch.launch()
                    ctx.check()
                    assert torch.equal(jobs[0][2], d_m), what
                    assert crt or torch.equal(jobs[1][2], d_c), what
                    batch.destroy()
            ctx.set_kernel_config(limbs, crt, 0)
            ctx.set_kernel_window(limbs, crt, 0)
    finally:
        ctx.set_batch_direct_max(256)
    ks.free()


@pytest.mark.parametrize("nbits", (2048, 3072, 4096, 6144, 8192))
def test_all_ones_primes_blinded(env, nbits):
    """Few chunks to many: each lane count of the blinded kernels."""
    import torch

    P, ctx = env
    p, q = _primes(nbits // 2)
    N = p * q
    ks = ctx.keyset_from_primes(nbits, 65537, _limbs([p], nbits // 2), _limbs([q], nbits // 2))
    rng = np.random.default_rng(nbits + 1)
    m = _operands(N, nbits, rng)
    r = [1, 2, N - 1, N - 2, (N >> 1) + 1, N >> 32, *(int.from_bytes(rng.bytes(nbits // 8), "little") % N
                                                     for _ in range(len(m) - 6))]
    star = _device([pow(x * y, 65537, N) for x, y in zip(m, r)], nbits)
    cr = _device([pow(y, 65537, N) for y in r], nbits)
    d_m = _device(m, nbits)
    for copies in (1, 50, 130, 700):
        got = ctx.decrypt_blinded(ks, star.repeat(copies, 1), cr.repeat(copies, 1), use_crt=True)
        assert torch.equal(got, d_m.repeat(copies, 1)), copies
    assert torch.equal(ctx.decrypt_blinded(ks, star, cr), d_m)  # inverse, product and full d
    a, b = ctx.encrypt_blinded(ks, d_m, _device(r, nbits))
    assert torch.equal(a, star) and torch.equal(b, cr)
    ctx.check()
    ks.free()


@pytest.mark.parametrize("nbits", (4096, 8192))
def test_all_ones_primes_four_residues(env, nbits):
    import torch

    P, ctx = env
    primes = _primes(nbits // 4, 4)
    N = primes[0] * primes[1] * primes[2] * primes[3]
    ks = ctx.keyset_from_primes_multi(nbits, 4, 65537, np.concatenate([_limbs([x], nbits // 4) for x in primes], axis=1))
    m = _operands(N, nbits, np.random.default_rng(nbits + 2))
    m += [x - 1 for x in primes] + [N - x for x in primes] + list(primes)
    d_m, d_c = _device(m, nbits), _device([pow(x, 65537, N) for x in m], nbits)
    assert torch.equal(ctx.encrypt_chunks(ks, d_m), d_c)
    limbs = nbits // 128
    for tpi, form in P.kernel_configs(limbs, True):
        ctx.set_kernel_config(limbs, True, tpi, form)
        assert torch.equal(ctx.decrypt_chunks(ks, d_c, use_crt=True), d_m), (tpi, form)
    ctx.set_kernel_config(limbs, True, 0)
    ctx.check()
    ks.free()


@pytest.mark.parametrize("nbits,sizes", [(2048, (1, 500, 700, 1300, 2500, 3700, 5000)),
                                         (3072, (1, 250, 700, 1300, 2600, 4000, 6000)),
                                         (4096, (1, 290, 320, 700, 1400, 2056, 3000))])
def test_choice_by_size_equals_pinned_geometry(env, nbits, sizes):
    import torch

    P, ctx = env
    pinned = P.Context(0)
    ks_a, ks_p = ctx.keygen(3, nbits, 65537, 61), pinned.keygen(3, nbits, 65537, 61)
    lanes = {False: set(), True: set()}
    for limbs, crt in ((nbits // 32, False), (nbits // 64, True)):
        pinned.set_kernel_config(limbs, crt, *pinned.get_kernel_config(limbs, crt))
    for n in sizes:
        m = _chunks_below(n, nbits, n)
        c = ctx.encrypt_chunks(ks_a, m)
        assert torch.equal(c, pinned.encrypt_chunks(ks_p, m)), n
        for crt in (False, True):
            lanes[crt].add(ctx.get_call_config(ks_a, crt, n)[0])
            assert torch.equal(ctx.decrypt_chunks(ks_a, c, use_crt=crt), m), (n, crt)
    ctx.check()
    assert all(len(v) > 1 for v in lanes.values()), lanes
    for ks in (ks_a, ks_p):
        ks.free()
    pinned.close()
