"""The lane count chosen from a call's size: at sizes on both sides of every
change of lanes, and for uneven keys, the result is the one of the pinned
geometry, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ctx():
    import paper_2111_11924_gb300 as P

    return P.Context(0)


def _message_chunks(n, nbits, seed):
    import torch

    raw = np.zeros((n, nbits // 8), np.uint8)
    raw[:, :-1] = np.random.default_rng(seed).integers(0, 256, (n, nbits // 8 - 1), dtype=np.uint8)
    return torch.from_numpy(raw.view(np.int32)).cuda()


# 1024 bits: 32-limb full width (4, 8, 16 lanes), 16-limb residues (2, 4, 8 lanes).  The lane count changes
# where the warps pass one or two per scheduler (608): 1216, 2432, 4864 exponentiations and their neighbours.
SIZES = (1, 2, 3, 31, 607, 608, 609, 1215, 1217, 1823, 2431, 2433, 3649, 4863, 4865, 7297, 9729)


@pytest.mark.parametrize("K", (1, 3, 16))
def test_size_rule_equals_pinned_geometry(K):
    import torch

    nbits = 1024
    auto, pinned = _ctx(), _ctx()
    ks_a, ks_p = auto.keygen(K, nbits, 65537, 91), pinned.keygen(K, nbits, 65537, 91)
    pinned.set_kernel_config(32, False, 4, 1)
    pinned.set_kernel_config(16, True, 2, 0)
    for n in SIZES:
        m = _message_chunks(n, nbits, n)
        c = auto.encrypt_chunks(ks_a, m)
        assert torch.equal(c, pinned.encrypt_chunks(ks_p, m)), ("encrypt", n)
        assert torch.equal(auto.decrypt_chunks(ks_a, c), m), ("decrypt", n)
        assert torch.equal(auto.decrypt_chunks(ks_a, c, use_crt=True), m), ("crt", n)
        idx = torch.from_numpy(np.random.default_rng(n).integers(0, K, n, dtype=np.int32)).cuda()
        ci = auto.encrypt_chunks(ks_a, m, key_idx=idx)
        assert torch.equal(ci, pinned.encrypt_chunks(ks_p, m, key_idx=idx)), ("encrypt idx", n)
        assert torch.equal(auto.decrypt_chunks(ks_a, ci, key_idx=idx), m), ("decrypt idx", n)
        assert torch.equal(auto.decrypt_chunks(ks_a, ci, use_crt=True, key_idx=idx), m), ("crt idx", n)
        r = _message_chunks(n, nbits, n + 1)
        star, cr = auto.encrypt_blinded(ks_a, m, r)
        assert torch.equal(auto.decrypt_blinded(ks_a, star, cr, use_crt=True), m), ("blinded", n)
    auto.check()
    pinned.check()


def test_size_rule_in_a_mixed_batch():
    import torch

    from paper_2111_11924_gb300 import pmkrsa

    ctx = _ctx()
    jobs, expect = [], []
    for i, (nbits, n, op) in enumerate(((512, 5, 0), (1024, 700, 1), (1024, 1300, 2), (2048, 40, 1),
                                        (2048, 900, 2), (512, 3000, 2))):
        ks = ctx.keygen(3, nbits, 65537, 17 + i)
        m = _message_chunks(n, nbits, i)
        c = ctx.encrypt_chunks(ks, m)
        src, want = (m, c) if op == 0 else (c, m)
        jobs.append((ks, src, torch.zeros_like(src), (pmkrsa.OP_ENCRYPT, pmkrsa.OP_DECRYPT, pmkrsa.OP_DECRYPT_CRT)[op]))
        expect.append(want)
    batch = ctx.batch(jobs)
    batch.launch()
    ctx.check()
    for (_, _, out, op), want in zip(jobs, expect):
        assert torch.equal(out, want), op
